"""Kernels that share work by size: the wide tensor-core reaction M2L (float32,
p = 11 .. 14), the charges' columns in P2M and L2P on both sides of their
thresholds, and the sort at the edges of its blocks."""
import numpy as np
import pytest

import oracle
from paper_1908_10863_gb300 import LayeredFMM, workloads

pytestmark = pytest.mark.gpu


# the float32 form's difference from FP64 at these orders is float32 arithmetic
# (3e-7 to 7e-7 in the potential, 2.5e-6 in the field): twice that
@pytest.mark.parametrize("p,n", [(11, 3000), (12, 20000), (13, 3000), (14, 20000)])
def test_wide_reaction_against_fp64(p, n):
    w = workloads.config2(n)
    Q = np.stack([w.q, w.q[::-1], np.abs(w.q)])
    out = {}
    for precision in (0, 1):
        with LayeredFMM(w.d, w.eps, p, precision=precision) as f:
            f.build(w.xyz, w.layer)
            out[precision] = f.evaluate(Q)
            one = f.evaluate(Q[1])[0]
            st = f.stats()
        assert st["reaction_keys"] > 0 and st["timeouts"] == 0
        assert oracle.err2(out[precision][0][1], one) < (1e-13, 1e-6)[precision]
    for r in range(3):
        assert oracle.err2(out[0][0][r], out[1][0][r]) < 1.5e-6
        assert oracle.err2(out[0][1][r], out[1][1][r]) < 5e-6


# one vector of n charges takes shared columns up to 19,455 (FP64) and 77,823
# (float32) charges, two vectors of them a thread per charge; the sums differ in
# order only
@pytest.mark.parametrize("precision,n,p", [(0, 19455, 4), (0, 10001, 10), (1, 77823, 6), (1, 40001, 10)])
def test_columns_shared_or_not(precision, n, p):
    w = workloads.config2(n)
    with LayeredFMM(w.d, w.eps, p, precision=precision) as f:
        f.build(w.xyz, w.layer)
        phi, E = f.evaluate(w.q)
        phi2, E2 = f.evaluate(np.stack([w.q, w.q]))
    tol = (1e-13, 1e-6)[precision]
    assert oracle.err2(phi, phi2[0]) < tol and oracle.err2(E, E2[1]) < 5 * tol


# one key more or less than full blocks and rounds; order of input does not matter
@pytest.mark.parametrize("n", [256, 257, 32768, 32769, 262145])
def test_order_of_charges(n):
    w = workloads.config2(n)
    s = np.random.default_rng(n).permutation(n)
    with LayeredFMM(w.d, w.eps, 3, precision=0) as f:
        f.build(w.xyz, w.layer)
        phi, E = f.evaluate(w.q)
        f.build(w.xyz[s], w.layer[s])
        phis, Es = f.evaluate(w.q[s])
    assert oracle.err2(phi[s], phis) < 1e-13 and oracle.err2(E[s], Es) < 1e-12
