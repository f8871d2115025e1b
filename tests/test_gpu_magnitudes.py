"""Charges of very different size, judged where the small ones are: the far
field's operands share one scale per level (float16 pieces in the float32 form,
63-bit digits in the FP64 form), so an error norm over all charges would show
only the large ones.  And charges whose digits are alike in every box."""
import numpy as np
import pytest

import oracle
from paper_1908_10863_gb300 import LayeredFMM, workloads

pytestmark = pytest.mark.gpu

# FP64 sums of a few thousand terms and the digits' 2^-63 of a level's largest
# multipole; float32: ten roundings of 6e-8 at full size, in each of the three
# evaluations compared.  A charge's potential falls off as 1/r only, so the
# largest charge's is within 2^6 of full size everywhere, and every part of the
# domain has to meet these by itself.
BOUND = {0: 1e-13, 1: 4e-6}


def _cells(xyz, k=8):
    lo, hi = xyz.min(0), xyz.max(0)
    c = np.minimum(((xyz - lo) / (hi - lo) * k).astype(int), k - 1)
    return (c[:, 0] * k + c[:, 1]) * k + c[:, 2]


def _worst_cell(diff, ref, cells):
    num, den = np.bincount(cells, diff ** 2), np.bincount(cells, ref ** 2)
    return np.sqrt(num[den > 0] / den[den > 0]).max()


@pytest.mark.parametrize("precision,p", [(0, 10), (0, 14), (1, 10), (1, 14)])
@pytest.mark.parametrize("large", [1e7, 1e12])
def test_one_large_charge(precision, p, large):
    w = workloads.config2(6000)
    a, b = np.zeros(w.n), w.q.copy()
    a[17], b[17] = large, 0.0
    with LayeredFMM(w.d, w.eps, p, precision=precision, leaf_cap=15) as f:
        f.build(w.xyz, w.layer)
        phi, _ = f.evaluate(np.stack([a + b, a, b]))
        assert f.stats()["timeouts"] == 0
    e = _worst_cell(phi[0] - phi[1] - phi[2], phi[0], _cells(w.xyz))
    print("precision %d p=%d: worst cell %.2e" % (precision, p, e))
    assert e < BOUND[precision]


@pytest.mark.parametrize("precision,p", [(0, 10), (1, 10)])
def test_layers_of_different_size(precision, p):
    w = workloads.config2(6000)
    a, b = np.where(w.layer == 0, w.q, 0.0), np.where(w.layer == 0, 0.0, 3e-7 * w.q)
    with LayeredFMM(w.d, w.eps, p, precision=precision) as f:
        f.build(w.xyz, w.layer)
        phi, E = f.evaluate(np.stack([a + b, a, b]))
    for l in range(3):
        at = w.layer == l
        e = (oracle.err2(phi[0][at], (phi[1] + phi[2])[at]), oracle.err2(E[0][at], (E[1] + E[2])[at]))
        print("precision %d layer %d: %.2e %.2e" % (precision, l, *e))
        assert e[0] < BOUND[precision] and e[1] < 10 * BOUND[precision]


# charges on a lattice, the same in every leaf: all sources of a tile have the
# same multipoles, and with 1/511, 1/3 and 255/511 their digits repeat
@pytest.mark.parametrize("p", [4, 10, 15])
@pytest.mark.parametrize("eps", [(1.0,), (1.0, 5.0, 10.0)])
def test_digits_alike_in_every_box(p, eps):
    k = 16
    g = (np.arange(k) + 0.3) / k
    x, y, z = (v.ravel() for v in np.meshgrid(g, g, g, indexing="ij"))
    d = [] if len(eps) == 1 else [-0.25, -0.5]
    xyz = np.column_stack([x, y, z - 0.9])
    layer = np.zeros(len(x), np.int32)
    for v in d:
        layer += xyz[:, 2] < v
    one = np.ones(len(x))
    S = (1.0 / 511, 1.0 / 3, 255.0 / 511)
    with LayeredFMM(d, list(eps), p, leaf_cap=2) as f:
        f.build(xyz, layer)
        phi, _ = f.evaluate(np.stack([one] + [s * one for s in S]))
        st = f.stats()
    assert st["m2l_free"] > 0 and st["timeouts"] == 0
    for s, v in zip(S, phi[1:]):
        # sums of 4,096 positive terms in two orders: 4,096 half ulps at most
        assert np.max(np.abs(v / s - phi[0]) / np.abs(phi[0])) < 5e-13
