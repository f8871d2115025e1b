"""FP64 reaction M2L by digit products on the tensor cores: orders at the edges
of its chunks and row parts against the oracle; linearity, to FP64 rounding,
over magnitudes and between charges of very different size; non-finite charges."""
import numpy as np
import pytest

import oracle
from paper_1908_10863_gb300 import LayeredFMM, workloads

pytestmark = pytest.mark.gpu

# truncation errors of this workload by order (geometric in p), with a margin of two
ORDERS = [(1, 3e-2), (4, 1.2e-3), (5, 5e-4), (7, 7e-5), (9, 1e-5), (12, 1e-6), (14, 2.1e-7)]


@pytest.mark.parametrize("p,tol", ORDERS)
def test_orders_match_oracle(p, tol):
    w = workloads.paper_p4()
    t = workloads.subsample(w.n, 200)
    with LayeredFMM(w.d, w.eps, p, precision=0) as f:
        f.build(w.xyz, w.layer)
        phi, E = f.evaluate(w.q)
        assert f.stats()["reaction_keys"] > 0
    ref, refE = oracle.direct(w.d, w.eps, w.xyz, w.layer, w.q, targets=t, mode=oracle.MODE_IMAGES)
    e = oracle.err2(ref, phi[t]), oracle.err2(refE, E[t])
    print("p=%d: Err2 %.2e %.2e" % (p, *e))
    assert e[0] < tol and e[1] < 10 * tol


# FP64 sums of a few thousand terms, and the digits' 2^-63 of the largest
# table value and multipole: below 1e-13 of the result
ROUND = 1e-13


@pytest.mark.parametrize("n,p", [(3000, 10), (20000, 10), (3000, 13)])
def test_superposition_and_scaling(n, p):
    w = workloads.config2(n)
    a, b = w.q, np.where(w.layer == 0, 1.0, 3e-7) * w.q[::-1]
    with LayeredFMM(w.d, w.eps, p, precision=0) as f:
        f.build(w.xyz, w.layer)
        phi, E = f.evaluate(np.stack([a + b, a, b, 3.7e-120 * a, 1.3e90 * a]))
        one, _ = f.evaluate(a)
        assert f.stats()["timeouts"] == 0
    assert oracle.err2(phi[0], phi[1] + phi[2]) < ROUND and oracle.err2(E[0], E[1] + E[2]) < ROUND
    assert oracle.err2(phi[1], phi[3] / 3.7e-120) < ROUND and oracle.err2(phi[1], phi[4] / 1.3e90) < ROUND
    assert oracle.err2(phi[1], one) < ROUND


def test_nonfinite_device_charge_stays_visible():
    import torch
    w = workloads.config2(3000)
    with LayeredFMM(w.d, w.eps, 6, precision=0) as f:
        f.build(w.xyz, w.layer)
        for bad in (np.nan, np.inf):
            q = w.q.copy()
            q[17] = bad
            qd = torch.tensor(q, device="cuda")
            phi = torch.zeros(w.n, dtype=torch.float64, device="cuda")
            f.evaluate_device(qd, phi)
            torch.cuda.synchronize()
            # the charge reaches every target, through the near field or an expansion
            assert not np.isfinite(phi.cpu().numpy()[np.arange(w.n) != 17]).any()
