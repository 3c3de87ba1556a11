"""FP64 results keep the accuracy of FP64 sums where the operands of a contraction span many
orders of magnitude: orbitals whose integrals, amplitudes and vectors fall off by up to 10^-3
each, CNTO vectors with weak orbitals, vectors that are not finite.

The FP64 pipe's sums are the reference.  Scaling orbital p by s_p scales every term of an
output element by the same product of its own orbitals' factors, so that FP64 sums keep the
relative accuracy of each element's terms: the elements are compared divided by that product,
each against the largest of its array.  Bound: sums of K <= 2000 products in any order differ
by at most 2 K 2^-53 < 5e-13 of their terms' magnitudes, which cancel by less than a factor of
20 in the largest element of these random sums (about K^(1/2) of K terms are left).
"""
import numpy as np
import pytest

from gpu_common import Case, run_all

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
TOL = 1e-11


def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _fall_off(c, decades):
    """Scale orbital p of a Case by s_p, 1 .. 10^-decades in a mixed order."""
    NO, NV, no, nv, _ = c.dims
    def factors(n, seed):
        return 10.0 ** (-decades * np.random.default_rng(seed).permutation(n) / max(1, n - 1))
    so, sv = factors(NO, 5), factors(NV, 6)
    so[:no], sv[:nv] = factors(no, 7), factors(nv, 8)
    s = np.concatenate([so, sv])
    y, st = c.sys, c.st
    y.chol = y.chol * s[:, None] * s[None, :]
    y.t1 = y.t1 * sv[:, None] * so[None, :]
    d = so[:no, None, None, None] * sv[None, :nv, None, None] * so[None, None, :, None] * sv[None, None, None, :]
    y.t2c, y.t2x, c.lam2 = y.t2c * d, y.t2x * d, c.lam2 * d
    c.lam1 = c.lam1 * sv[:, None] * so[None, :]
    st.R1, st.L1 = (x * sv[None, :, None] * so[None, None, :] for x in (st.R1, st.L1))
    st.R2, st.L2 = (x * d[None] for x in (st.R2, st.L2))
    return c, {"o1": sv[:, None] * so[None, :], "o2": d, "D": s[:, None] * s[None, :]}


@pytest.mark.parametrize("decades", [0.0, 1.0, 3.0])
@pytest.mark.parametrize("dims", [(6, 24, 4, 8, 72), (7, 40, 3, 32, 60), (5, 60, 5, 50, 40)])
def test_weak_orbitals(dims, decades):
    _cuda()
    c, factor = _fall_off(Case(*dims, nstates=1, t2_norm=0.3), decades)
    factor.update(rho1=factor["o1"], sig1=factor["o1"], rho2=factor["o2"], sig2=factor["o2"])
    got = run_all(c, c.context(params={"fp64_tc_from": 1}))
    ref = run_all(c, c.context(params={"fp64_tc_from": 2000}))
    for k in got:
        f = factor.get(k, factor["D"])
        err, size = np.max(np.abs(got[k] - ref[k]) / f), np.max(np.abs(ref[k]) / f)
        assert err < TOL * size, (k, err / size)


def test_one_large_element_outside_the_products():
    """One Cholesky element between two inactive orbitals sets the largest magnitude of the
    factors and meets no active index in the triples' integrals."""
    _cuda()
    c = Case(7, 40, 3, 32, 60, nstates=1, t2_norm=0.3)
    p = 6  # an occupied orbital that is not active
    c.sys.chol = np.array(c.sys.chol)
    c.sys.chol[0, p, p] = 1e7
    c.sys.t1 = np.zeros_like(c.sys.t1)  # (T1 would mix it into the active blocks)
    got = run_all(c, c.context(params={"fp64_tc_from": 1}))
    ref = run_all(c, c.context(params={"fp64_tc_from": 2000}))
    for k in ("o1", "o2"):
        assert np.linalg.norm(got[k] - ref[k]) < TOL * np.linalg.norm(ref[k]), k


@pytest.mark.parametrize("NO,NV,decades", [(9, 40, 0.0), (9, 40, 1.0), (9, 40, 5.0), (39, 60, 4.0), (130, 9, 4.0)])
def test_weak_orbitals_of_the_cnto_matrices(NO, NV, decades):
    """|M_ij - sum| <= 2 K 2^-53 (M_ii M_jj)^(1/2) by Cauchy-Schwarz, K = N_V^2 N_O products."""
    _cuda()
    from paper_2202_08612_gb300 import cnto
    rng = np.random.default_rng(NO * NV)
    fo = 10.0 ** (-decades * rng.permutation(NO) / (NO - 1))
    fv = 10.0 ** (-decades * rng.permutation(NV) / (NV - 1))
    R1 = rng.normal(size=(NV, NO)) * fv[:, None] * fo[None, :]
    f = (fv[:, None] * fo[None, :]).reshape(-1)
    P = rng.normal(size=(NV * NO, NV * NO))
    R2 = ((P + P.T) * f[:, None] * f[None, :]).reshape(NV, NO, NV, NO)
    X, Y = R2.transpose(1, 0, 2, 3).reshape(NO, -1), R2.reshape(NV, -1)
    dd = np.einsum("aiai->ai", R2)
    Mo = R1.T @ R1 + 0.5 * X @ X.T + 0.5 * np.diag((dd * dd).sum(0))
    No = R1 @ R1.T + 0.5 * Y @ Y.T + 0.5 * np.diag((dd * dd).sum(1))
    M, N = cnto.cnto_matrices(torch.from_numpy(R1).cuda(), torch.from_numpy(R2).cuda())
    for got, ref, K in ((M.cpu().numpy(), Mo, NV * NV * NO), (N.cpu().numpy(), No, NO * NO * NV)):
        d = np.sqrt(np.diag(ref))
        assert np.max(np.abs(got - ref) / (d[:, None] * d[None, :])) < 2 * K * 2.0 ** -53


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_values_that_are_not_finite(value):
    """The same outputs are infinite, NaN and finite as in FP64 arithmetic, in the call that
    meets such a vector and (all finite) in the next one."""
    _cuda()
    c = Case(7, 40, 3, 32, 60, nstates=1, t2_norm=0.3)
    R2 = np.array(c.st.R2)
    R2[0, 1, 2, 0, 35] = value
    outs = []
    for start in (1, 2000):
        g = c.context(params={"fp64_tc_from": start})
        for x in (R2, c.st.R2):
            r1, r2 = c.empty_dev(c.st.R1.shape), c.empty_dev(c.st.R2.shape)
            g.jacobian_right(c.st.omega, c.to_dev(c.st.R1), c.to_dev(x), r1, r2)
            outs += [c.host(r1), c.host(r2)]
    for x, y in zip(outs[:4], outs[4:]):
        assert np.array_equal(np.isnan(x), np.isnan(y)) and np.array_equal(np.isposinf(x), np.isposinf(y))
    assert not np.isfinite(outs[1]).all() and np.isfinite(outs[3]).all()


@pytest.mark.parametrize("decades", [0.0, 4.0])
def test_outputs_over_their_inputs(decades):
    """rho2 and sigma2 into the vector's own array, of a call that runs once and of one that
    runs again on the FP64 pipe after it."""
    _cuda()
    c, _ = _fall_off(Case(7, 40, 3, 32, 60, nstates=2, t2_norm=0.3), decades)
    ref = c.context(params={"fp64_tc_from": 2000})
    for call, X1, X2 in (("jacobian_right", c.st.R1, c.st.R2), ("jacobian_left", c.st.L1, c.st.L2)):
        g = c.context(params={"fp64_tc_from": 1})
        x1, x2 = c.to_dev(X1), c.to_dev(X2)
        y1, y2 = c.empty_dev(X1.shape), c.empty_dev(X2.shape)
        getattr(ref, call)(c.st.omega, x1, x2, y1, y2)
        z1 = c.empty_dev(X1.shape)
        getattr(g, call)(c.st.omega, x1, x2, z1, x2)
        assert np.linalg.norm(c.host(x2) - c.host(y2)) < TOL * np.linalg.norm(c.host(y2))
        assert np.linalg.norm(c.host(z1) - c.host(y1)) < TOL * np.linalg.norm(c.host(y1))


def test_weak_rows_stay_on_the_tensor_cores():
    """A vector whose elements on some inactive virtual orbitals are 10^-9 of the others makes
    weak rows in Upsilon's factors, which have scales of their own: no FP64 build is launched,
    and the parts of rho that come from those orbitals alone are as on the FP64 pipe."""
    _cuda()
    c = Case(7, 60, 3, 32, 60, nstates=1, t2_norm=0.3)
    c.st.R1, c.st.R2 = np.array(c.st.R1), np.array(c.st.R2)
    c.st.R1[0, 40:50] *= 1e-9
    c.st.R2[...] = 0.0
    outs = []
    for start in (1, 2000):
        g = c.context(params={"fp64_tc_from": start})
        r1, r2 = c.empty_dev(c.st.R1.shape), c.empty_dev(c.st.R2.shape)
        g.profile(False)
        g.jacobian_right(c.st.omega, c.to_dev(c.st.R1), c.to_dev(c.st.R2), r1, r2)
        names = set(g.kernel_stats())
        assert ("triples_build_kernel" in names) == (start == 2000), names
        outs.append((c.host(r1), c.host(r2)))
    for x, y in zip(*outs):
        assert np.linalg.norm(x - y) < 1e-12 * np.linalg.norm(y)


@pytest.mark.parametrize("decades", [0.0, 4.0])
def test_host_arrays(decades):
    """Inputs and outputs in host memory, of calls that run once and of ones that run again."""
    _cuda()
    c, factor = _fall_off(Case(7, 40, 3, 32, 60, nstates=2, t2_norm=0.3), decades)
    ref, g = c.context(params={"fp64_tc_from": 2000}), c.context(params={"fp64_tc_from": 1}, device=False)
    for call, X1, X2 in (("jacobian_right", c.st.R1, c.st.R2), ("jacobian_left", c.st.L1, c.st.L2)):
        y1, y2 = c.empty_dev(X1.shape), c.empty_dev(X2.shape)
        getattr(ref, call)(c.st.omega, c.to_dev(X1), c.to_dev(X2), y1, y2)
        for _ in range(2):
            z1, z2 = np.full(X1.shape, 7.0), np.full(X2.shape, 7.0)
            getattr(g, call)(c.st.omega, np.ascontiguousarray(X1), np.ascontiguousarray(X2), z1, z2)
            for x, y, f in ((z1, c.host(y1), factor["o1"]), (z2, c.host(y2), factor["o2"])):
                assert np.max(np.abs(x - y) / f) < TOL * np.max(np.abs(y) / f), call
