"""Reaction M2L in the rotated frame (FP64 form, and float32 off the tensor
cores) against the oracle: orders on both sides of its staging widths (p = 10
and 11) and of the former limit of keyed orders (p = 15 and 16)."""
import numpy as np
import pytest

import oracle
from paper_1908_10863_gb300 import LayeredFMM, workloads
from paper_1908_10863_gb300.lfmm import OPT_TENSOR_CORES

pytestmark = pytest.mark.gpu

# truncation errors of this workload by order (geometric in p), with a margin
# of two; float32 arithmetic adds about 5e-7
CASES = [(0, 2, 1e-2), (0, 10, 5e-6), (0, 11, 3e-6), (0, 15, 1.2e-7), (0, 16, 6e-8), (0, 20, 4e-10),
         (1, 10, 6e-6), (1, 11, 3e-6), (1, 14, 1.2e-6)]


@pytest.mark.parametrize("precision,p,tol", CASES)
def test_orders_match_oracle(precision, p, tol):
    w = workloads.paper_p4()
    t = workloads.subsample(w.n, 200)
    Q = np.stack([w.q, w.q[::-1]])
    with LayeredFMM(w.d, w.eps, p, precision=precision) as f:
        f.set_option(OPT_TENSOR_CORES, 0)
        f.build(w.xyz, w.layer)
        phi, E = f.evaluate(Q)
        st = f.stats()
    assert st["m2l_reaction"] > 0 and st["reaction_keys"] > 0
    for r in range(2):
        ref, refE = oracle.direct(w.d, w.eps, w.xyz, w.layer, Q[r], targets=t, mode=oracle.MODE_IMAGES)
        e = oracle.err2(ref, phi[r][t]), oracle.err2(refE, E[r][t])
        print("precision %d p=%d: Err2 %.2e %.2e" % (precision, p, *e))
        assert e[0] < tol and e[1] < 10 * tol
