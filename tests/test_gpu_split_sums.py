"""Reductions split over blocks, against 64-bit-mantissa (or longer) sums: the pieces of one
product are added up before they meet the output, so the singles of sigma, sums of some ten
products, are as exact as with reductions that are not split ("bstc_fill" 0).

The error of a call is a random walk of roundings; over the systems below the mean of its
logarithm varies by about 0.1 (the spread of one call, 30 %, over the square root of ten), so
1.35 between the two forms is three such deviations."""
import os
import sys
import types

import numpy as np
import pytest

from gpu_common import Case

pytestmark = pytest.mark.gpu


def _long_oracle():
    """The oracle's equations in numpy's longest floating type."""
    path = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "oracle", "mlcc3_oracle.py")
    src = open(path).read().replace("np.float64", "np.longdouble")
    src = src.replace("np.zeros(", "_zeros(").replace("np.eye(", "_eye(")
    m = types.ModuleType("long_oracle")
    m._zeros = lambda shape, dtype=np.longdouble: np.zeros(shape, dtype=dtype)
    m._eye = lambda n: np.eye(n, dtype=np.longdouble)
    sys.modules["long_oracle"] = m  # (its dataclasses look their module up)
    exec(compile(src, "long_oracle", "exec"), m.__dict__)
    return m


def test_sigma_singles_are_as_exact_as_unsplit_sums():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    O = _long_oracle()
    logs = {4: [], 0: []}
    for seed in range(10):
        c = Case(*[(6, 24, 4, 8, 72), (5, 30, 3, 9, 90)][seed % 2], nstates=1, seed=500 + seed, t2_norm=0.3)
        o, st = O.make_ctx(c.sys), c.st
        ref, _ = O.jacobian_left(o, np.longdouble(st.omega[0]), st.L1[0].astype(np.longdouble), O.to_full(o, st.L2[0]))
        for fill, out in logs.items():
            g = c.context(params={"bstc_fill": fill, "fp64_tc_from": 2000})
            s1, s2 = c.empty_dev(st.L1.shape), c.empty_dev(st.L2.shape)
            g.jacobian_left(st.omega, c.to_dev(st.L1), c.to_dev(st.L2), s1, s2)
            d = c.host(s1)[0].astype(np.longdouble) - ref
            out.append(float(np.log(np.sqrt(np.sum(d * d) / np.sum(ref * ref)))))
    assert np.mean(logs[4]) < np.mean(logs[0]) + np.log(1.35), np.exp([np.mean(logs[4]), np.mean(logs[0])])
