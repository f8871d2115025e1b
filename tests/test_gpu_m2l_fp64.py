"""FP64 free M2L by digit products on the tensor cores: against the oracle by
order, and to rounding by superposition and scaling (every evaluation has its
own digit scale, so an inexact product would break both)."""
import numpy as np
import pytest

import oracle
from paper_1908_10863_gb300 import LayeredFMM, workloads

pytestmark = pytest.mark.gpu

# FP64 sums of a few thousand terms, and the digits' 2^-63 of the largest
# multipole of a level: below 1e-13 of the result
ROUND = 1e-13


def _eval(w, p, Q, leaf_cap=40):
    with LayeredFMM(w.d, w.eps, p, leaf_cap=leaf_cap) as f:
        f.build(w.xyz, w.layer)
        phi, E = f.evaluate(Q)
        st = f.stats()
    assert st["m2l_free"] > 0 and st["timeouts"] == 0
    return phi, E


# (p + 1)^2 at the edges of the K chunks and steps (9, 36, 49, 64, 121) and of
# the output halves (144, 256); bounds: twice the truncation errors by order
@pytest.mark.parametrize("p,tol", [(2, 1e-2), (5, 6e-4), (6, 2e-4), (7, 8e-5), (10, 5e-6), (11, 3e-6), (15, 1.2e-7)])
def test_orders_match_oracle(p, tol):
    w = workloads.paper_p4()
    t = workloads.subsample(w.n, 200)
    phi, E = _eval(w, p, w.q)
    ref, refE = oracle.direct(w.d, w.eps, w.xyz, w.layer, w.q, targets=t, mode=oracle.MODE_IMAGES)
    assert oracle.err2(ref, phi[t]) < tol and oracle.err2(refE, E[t]) < 10 * tol


# 700 charges (leaves of 10, so that the tree has far pairs): merged tiles with a few targets each; 12,000 with leaves of 10:
# several full tiles per class
@pytest.mark.parametrize("n,p,cap", [(700, 10, 10), (700, 4, 10), (12000, 10, 10), (5000, 14, 10)])
def test_superposition_and_scaling(n, p, cap):
    w = workloads.config2(n)
    rng = np.random.default_rng(3)
    a, b = w.q, rng.uniform(0.0, 1.0, n) ** 8 * 1e-4
    phi, E = _eval(w, p, np.stack([a + b, a, b, a * 1e-200, a * 1e180]), cap)
    assert oracle.err2(phi[0], phi[1] + phi[2]) < ROUND and oracle.err2(E[0], E[1] + E[2]) < ROUND
    for r, s in ((3, 1e-200), (4, 1e180)):
        assert oracle.err2(phi[1], phi[r] / s) < ROUND and oracle.err2(E[1], E[r] / s) < ROUND


def test_single_sided_and_empty_offsets():
    # charges in two thin sheets: most offsets of a tile have no source
    rng = np.random.default_rng(4)
    n = 4000
    xyz = np.column_stack([rng.uniform(-1, 1, (n, 2)), np.where(np.arange(n) % 2, 0.3, -0.3) + rng.uniform(0, 1e-3, n)])
    lay = np.zeros(n, np.int32)
    q = rng.uniform(-1, 1, n)
    with LayeredFMM([], [1.0], 12) as f:
        f.build(xyz, lay)
        phi, E = f.evaluate(q)
    ref, refE = oracle.direct([], [1.0], xyz, lay, q, mode=oracle.MODE_FREE_ONLY)
    assert oracle.err2(ref, phi) < 1e-5 and oracle.err2(refE, E) < 1e-4
