"""Near field by lists of sources with image rules (FP64, and float32 with
reaction pairs): trees of one or a few boxes, so that every pair is a near
pair, against the oracle's exact image series."""
import numpy as np
import pytest

import oracle
from paper_1908_10863_gb300 import LayeredFMM, workloads

pytestmark = pytest.mark.gpu

# kappa = product of the middle layer's reflections: -0.22, 0.93, 0.95, -0.9, 0
# (one interface vanishes)
MEDIA = [(1.0, 5.0, 10.0), (1.0, 80.0, 2.0), (80.0, 1.0, 80.0), (1.0, 20.0, 4000.0), (1.0, 5.0, 5.0)]
# FP64: the rules reproduce the remainder to 2e-14, sums of a few hundred terms
# add rounding; float32: offsets of ~1 rounded at 6e-8 against pair distances
# of 0.04 and more (1.5e-6), twice that in the squared distances of the field
TOL = {0: (1e-11, 1e-11), 1: (5e-6, 1e-5)}


def _run(w, precision, cap, nrhs):
    q = np.stack([np.roll(w.q, 3 * r) for r in range(nrhs)])
    with LayeredFMM(w.d, w.eps, 4, precision=precision, leaf_cap=cap) as f:
        f.build(w.xyz, w.layer)
        phi, E = f.evaluate(q if nrhs > 1 else q[0])
        st = f.stats()
    return q, phi.reshape(nrhs, -1), E.reshape(nrhs, -1, 3), st


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n", [4, 31, 67, 259])  # boxes of 1 .. 65 charges: target slots and staged chunks part full
def test_one_box_per_layer_matches_images(precision, n):
    for eps in MEDIA:
        w = workloads.near_interface(n, delta=0.1, hmin=0.02, eps=eps)
        _, phi, E, st = _run(w, precision, 100000, 1)
        assert st["m2l_free"] == 0 and st["m2l_reaction"] == 0 and st["p2p_reaction"] > 0
        ref, refE = oracle.direct(w.d, w.eps, w.xyz, w.layer, w.q, mode=oracle.MODE_IMAGES)
        e = oracle.err2(ref, phi[0]), oracle.err2(refE, E[0])
        print("eps %s n=%d precision %d: Err2 %.2e %.2e" % (eps, n, precision, *e))
        assert e[0] < TOL[precision][0] and e[1] < TOL[precision][1]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nrhs", [2, 3, 9])  # partial batches of every launch width
def test_several_vectors_match_images(precision, nrhs):
    w = workloads.near_interface(150, delta=0.1, hmin=0.02)
    q, phi, E, _ = _run(w, precision, 100000, nrhs)
    for r in range(nrhs):
        ref, refE = oracle.direct(w.d, w.eps, w.xyz, w.layer, q[r], mode=oracle.MODE_IMAGES)
        assert oracle.err2(ref, phi[r]) < TOL[precision][0] and oracle.err2(refE, E[r]) < TOL[precision][1]


def test_wide_layout_keeps_its_accuracy():
    # rho many times the depth: no quadrature has to follow J0 here
    w = workloads.slab(300, half_width=50.0)
    _, phi, E, _ = _run(w, 0, 100000, 1)
    ref, refE = oracle.direct(w.d, w.eps, w.xyz, w.layer, w.q, mode=oracle.MODE_IMAGES)
    assert oracle.err2(ref, phi[0]) < 1e-11 and oracle.err2(refE, E[0]) < 1e-11
