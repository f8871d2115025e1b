"""LFMM_OPT_NEAR_TABLES = 0 takes the near-field reaction kernels by the
quadrature, in media whose automatic choice is the image sums too."""
import pytest

import oracle
from paper_1908_10863_gb300 import LayeredFMM, workloads
from paper_1908_10863_gb300.lfmm import OPT_NEAR_TABLES

pytestmark = pytest.mark.gpu


def test_quadrature_on_request():
    # a flat layout in one box per layer: lateral distances of many times the
    # depth, where the quadrature is off by parts in a million and the image
    # sums (good to 2e-14 per pair) are not
    w = workloads.slab(300, half_width=50.0)
    ref, _ = oracle.direct(w.d, w.eps, w.xyz, w.layer, w.q, mode=oracle.MODE_IMAGES)
    err = []
    with LayeredFMM(w.d, w.eps, 4, leaf_cap=100000) as f:
        f.build(w.xyz, w.layer)
        for use in (2, 0, 2):
            f.set_option(OPT_NEAR_TABLES, use)
            err.append(oracle.err2(ref, f.evaluate(w.q)[0]))
    print("Err2 %.2e by the automatic choice, %.2e by quadrature" % (err[0], err[1]))
    assert err[0] < 1e-11 and err[2] < 1e-11
    assert 1e-9 < err[1] < 1e-4


# float32: the quadrature in the kernels of one and of several vectors
@pytest.mark.parametrize("nrhs", [1, 3])
def test_float32_quadrature_on_request(nrhs):
    import numpy as np
    w = workloads.near_interface(2000, delta=0.1, hmin=0.02)
    Q = np.stack([np.roll(w.q, r) for r in range(nrhs)])
    out = {}
    for precision, use in ((0, 0), (1, 0), (1, 2)):
        with LayeredFMM(w.d, w.eps, 8, precision=precision) as f:
            f.set_option(OPT_NEAR_TABLES, use)
            f.build(w.xyz, w.layer)
            out[precision, use] = f.evaluate(Q)
            assert f.stats()["p2p_reaction"] > 0
    for use in (0, 2):
        for r in range(nrhs):  # float32 offsets of ~1 against distances of 0.04 and more
            assert oracle.err2(out[0, 0][0][r], out[1, use][0][r]) < 5e-6
            assert oracle.err2(out[0, 0][1][r], out[1, use][1][r]) < 2e-5
