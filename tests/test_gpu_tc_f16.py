"""Tensor-core free M2L and leaf L2L with float16 operand pieces: orders at the
edges of the K steps and chunks, and charges of very different magnitudes (the
pieces' scale follows the largest multipole), against the FP64 form."""
import numpy as np
import pytest

import oracle
from paper_1908_10863_gb300 import LayeredFMM, workloads

pytestmark = pytest.mark.gpu

# float32 arithmetic against FP64 at the same order: accumulation of 9 offsets
# per accumulator and of the near field, ~10 roundings of 6e-8 at full size
BOUND = 2e-6


def _both(w, p, q):
    out = []
    for precision in (0, 1):
        with LayeredFMM(w.d, w.eps, p, precision=precision) as f:
            f.build(w.xyz, w.layer)
            out.append(f.evaluate(q))
            st = f.stats()
    assert st["timeouts"] == 0 and st["m2l_free"] > 0
    return out


# (p + 1)^2 = 16, 25, 36, 49, 64, 121 | 144, 225 (wide): one and two chunks of
# 32 coefficients, a chunk with one of its two K steps, the last chunk nearly full
@pytest.mark.parametrize("p", [1, 3, 4, 5, 6, 7, 10, 11, 14])
def test_orders_match_fp64(p):
    w = workloads.config2(5001)
    (phi, E), (phi32, E32) = _both(w, p, w.q)
    assert oracle.err2(phi, phi32) < BOUND and oracle.err2(E, E32) < 10 * BOUND


# down to charges whose degree-12 multipoles (1e-13 of a charge in box units)
# are still normal float32 numbers
@pytest.mark.parametrize("scale", [1e-24, 1e-19, 1e25])
@pytest.mark.parametrize("p", [10, 12])
def test_magnitudes_match_fp64(p, scale):
    w = workloads.config2(6000)
    (phi, E), (phi32, E32) = _both(w, p, w.q * scale)
    assert oracle.err2(phi, phi32) < BOUND and oracle.err2(E, E32) < 10 * BOUND


def test_zero_charges_and_one_large():
    w = workloads.config2(6000)
    q = np.zeros(w.n)
    (_, _), (phi32, E32) = _both(w, 10, q)
    assert np.all(phi32 == 0.0) and np.all(E32 == 0.0)
    q[:] = w.q
    q[17] = 1e7  # one box's multipole dwarfs every other's
    (phi, E), (phi32, E32) = _both(w, 10, q)
    assert oracle.err2(phi, phi32) < BOUND and oracle.err2(E, E32) < 10 * BOUND


def test_vectors_have_their_own_scale():
    w = workloads.config2(6000)
    Q = np.stack([w.q * 1e-12, w.q[::-1] * 1e9, w.q])
    (phi, E), (phi32, E32) = _both(w, 10, Q)
    for r in range(3):
        assert oracle.err2(phi[r], phi32[r]) < BOUND and oracle.err2(E[r], E32[r]) < 10 * BOUND
