"""lfmm_evaluate_device returns once its work is enqueued, the first call of a
context included."""
import pytest

import oracle
from paper_1908_10863_gb300 import LayeredFMM, workloads

pytestmark = pytest.mark.gpu


# the digit form's orders (one and two halves) and the order above them, and float32
@pytest.mark.parametrize("precision,p", [(0, 10), (0, 12), (0, 16), (1, 10)])
@pytest.mark.parametrize("switched", [False, True])  # the form chosen before or after the build
def test_first_evaluation_does_not_wait(precision, p, switched):
    import torch
    w = workloads.config2(3000)
    q = torch.from_numpy(w.q).cuda()

    def context():
        f = LayeredFMM(w.d, w.eps, p, precision=(1 - precision if switched and p <= 14 else precision))
        f.build(w.xyz, w.layer)
        f.set_option(1, precision)
        return f

    with context() as f:  # (every kernel is loaded)
        ref, _ = f.evaluate(w.q)
    phi = torch.zeros_like(q)
    side = torch.cuda.Stream()
    with context() as f:
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            torch.cuda._sleep(1_000_000_000)  # ~0.5 s
            slept = torch.cuda.Event()
            slept.record()
        f.evaluate_device(q, phi, stream=side)
        busy = not slept.query()
        torch.cuda.synchronize()
        assert f.stats()["timeouts"] == 0
    assert busy, "the call waited for the stream"
    assert oracle.err2(ref, phi.cpu().numpy()) < (1e-13, 1e-6)[precision]
