"""LFMM_OPT_QUAD_NODES set at any point between build and evaluation: the
reaction M2L's tables follow the rule in force at the evaluation."""
import pytest

import oracle
from paper_1908_10863_gb300 import LayeredFMM, workloads
from paper_1908_10863_gb300.lfmm import OPT_QUAD_NODES

pytestmark = pytest.mark.gpu

# the same tables twice: sums of a few thousand FP64 terms in another order
# (float32: of float32 terms)
ROUND = {0: 1e-13, 1: 1e-6}


def _phi(w, precision, steps):
    """The potentials of the last evaluation; steps: "build", "evaluate" or a node count."""
    with LayeredFMM(w.d, w.eps, 8, precision=precision) as f:
        for s in steps:
            if s == "build":
                f.build(w.xyz, w.layer)
            elif s == "evaluate":
                phi, _ = f.evaluate(w.q)
            else:
                f.set_option(OPT_QUAD_NODES, s)
        assert f.stats()["reaction_keys"] > 0 and f.stats()["timeouts"] == 0
    return phi


@pytest.mark.parametrize("precision", [0, 1])
def test_nodes_changed_between_build_and_evaluation(precision):
    # (a product of reflections of 0.41; above 0.44 the rule is fixed)
    w = workloads.config2(3000, eps=(1.0, 4.5, 1.0))
    ref = {q: _phi(w, precision, (q, "build", "evaluate")) for q in (16, 128)}
    if precision == 0:  # 16 nodes are too few for this medium: the two rules can be told apart
        assert oracle.err2(ref[128], ref[16]) > 1e-10
    for q in (16, 128):  # fewer and more nodes than the default's 64
        assert oracle.err2(ref[q], _phi(w, precision, ("build", q, "evaluate"))) < ROUND[precision]
    # tables that an evaluation has made already
    assert oracle.err2(ref[128], _phi(w, precision, (16, "build", "evaluate", 128, "evaluate"))) < ROUND[precision]
    assert oracle.err2(ref[16], _phi(w, precision, (128, "build", "evaluate", 16, "evaluate"))) < ROUND[precision]


def test_nodes_changed_while_an_evaluation_is_queued():
    # the option waits for work that reads the rule; the evaluation keeps its own
    import torch
    w = workloads.config2(3000, eps=(1.0, 4.5, 1.0))
    ref = _phi(w, 0, ("build", "evaluate"))
    q = torch.from_numpy(w.q).cuda()
    phi = torch.zeros_like(q)
    side = torch.cuda.Stream()
    with LayeredFMM(w.d, w.eps, 8, precision=0) as f:
        f.build(w.xyz, w.layer)
        f.evaluate(w.q)
        f.build(w.xyz, w.layer)  # (tables to be made again; every buffer has its size)
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            torch.cuda._sleep(200_000_000)  # ~0.1 s
            f.evaluate_device(q, phi, stream=side)
        f.set_option(OPT_QUAD_NODES, 16)
        torch.cuda.synchronize()
    assert oracle.err2(ref, phi.cpu().numpy()) < ROUND[0]
