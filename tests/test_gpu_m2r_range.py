"""Float32 reaction M2L on the tensor cores where the operators leave float16's
range: thin middle layers of high permittivity, whose image series adds
hundreds to thousands of images at a fraction of a box apart, and media whose
reflections nearly vanish."""
import numpy as np
import pytest

import oracle
from paper_1908_10863_gb300 import LayeredFMM
from paper_1908_10863_gb300.lfmm import OPT_TENSOR_CORES

pytestmark = pytest.mark.gpu

# float32 arithmetic at the same order, ~10 roundings of 6e-8 at full size (as in
# the free M2L's comparison with FP64), of two forms; the field ten times that
BOUND = 4e-6


def _points(n, D):
    """Half the charges in a middle layer (-D, 0), half above it, up to 1.5."""
    rng = np.random.default_rng(5)
    m = n // 2
    z = np.concatenate([-D * rng.uniform(0.05, 0.95, m), rng.uniform(0.3, 1.5, n - m)])
    xyz = np.column_stack([rng.uniform(-1, 1, (n, 2)), z])
    return xyz, np.where(np.arange(n) < m, 1, 0).astype(np.int32), rng.uniform(-1, 1, n)


# largest image sums sum_n kappa^n / (2 + 2 n D / h) at h of a quarter: about 600
# and 6,000, twice that through an interface; and reflections of 5e-7
@pytest.mark.parametrize("p,D,eps", [(6, 2e-4, (1.0, 1e4, 1.0)), (10, 2e-4, (1.0, 1e4, 1.0)),
                                     (10, 2e-5, (1.0, 1e5, 1.0)), (13, 2e-4, (1.0, 1e4, 1.0)),
                                     (10, 0.2, (1.0, 1.000001, 1.0))])
@pytest.mark.parametrize("nrhs", [1, 3])
def test_operators_of_any_size(p, D, eps, nrhs):
    xyz, layer, q = _points(4000, D)
    Q = np.stack([np.roll(q, 7 * r) for r in range(nrhs)])
    out = {}
    # the same near field in both, so what differs is the M2L's engine
    for tc in (0, 1):
        with LayeredFMM([0.0, -D], eps, p, precision=1) as f:
            f.set_option(OPT_TENSOR_CORES, tc)
            f.build(xyz, layer)
            out[tc] = f.evaluate(Q)
            st = f.stats()
        assert st["reaction_keys"] > 0 and st["timeouts"] == 0
    (phi0, E0), (phi1, E1) = out[0], out[1]
    assert np.isfinite(phi1).all() and np.isfinite(E1).all()
    for r in range(nrhs):
        e = oracle.err2(phi0[r], phi1[r]), oracle.err2(E0[r], E1[r])
        print("p=%d D=%g eps %s: Err2 %.2e %.2e" % (p, D, eps, *e))
        assert e[0] < BOUND and e[1] < 10 * BOUND
