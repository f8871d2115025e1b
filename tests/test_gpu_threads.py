"""Contexts of different orders, sizes and media evaluated from several host
threads at once: launch limits are properties of the process, so no context may
lower what another is about to need."""
import threading

import numpy as np
import pytest

import oracle
from paper_1908_10863_gb300 import LayeredFMM, workloads

pytestmark = pytest.mark.gpu

# (precision, order, charges): every kernel whose shared memory follows the
# order, the quadrature or the geometry
SETS = [
    [(0, 4, 1500), (0, 10, 2500), (0, 15, 1200)],   # digit forms, P2M / L2P
    [(0, 16, 900), (0, 20, 1200), (0, 16, 1500)],   # rotated form, per-pair M2L
    [(1, 5, 1500), (1, 10, 3000), (1, 14, 2500)],   # float32
]


@pytest.mark.parametrize("members", SETS)
def test_contexts_from_several_threads(members):
    jobs, ref = [], []
    for i, (precision, p, n) in enumerate(members):
        w = workloads.config2(n, seed=i + 3)
        f = LayeredFMM(w.d, w.eps, p, precision=precision, leaf_cap=10 + 15 * i)
        f.build(w.xyz, w.layer)
        jobs.append((f, w, precision))
        ref.append(f.evaluate(w.q)[0])
    bad = []
    start = threading.Barrier(len(jobs))

    def work(i):
        f, w, precision = jobs[i]
        start.wait()
        try:
            for k in range(150):
                if k % 10 == 9:  # (the tables again)
                    f.build(w.xyz, w.layer)
                e = oracle.err2(ref[i], f.evaluate(w.q)[0])
                if not e < (1e-12, 1e-5)[precision]:
                    bad.append((i, k, e))
        except Exception as e:  # noqa: BLE001
            bad.append((i, k, str(e)))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for f, _, _ in jobs:
        f.close()
    assert not bad, bad[:5]
