"""Gradients registered again while a fused step that uses the old ones is
still to run: nothing but lc_register_optimizer's own wait keeps the step's
table as it was, since a stream of torch's own is not ordered with the
upload."""
import pytest

from tests.lc_harness import require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("engine", ["bulk", "threads"])
def test_optimizer_registered_again_behind_a_queued_step(engine):
    """Two steps with two sets of gradients, the first still queued behind
    other work when the second set is registered, against the same steps of
    a context that waits after each: weights and moments are the same bits."""
    torch = require_gpu()
    import paper_2609_27193_gb300 as P
    g = torch.Generator(device="cuda").manual_seed(3)
    sizes = [4096, 257, 100003]
    rand = lambda n, s: torch.randn(n, generator=g, device="cuda") * s
    base = [(rand(n, 0.02), rand(n, 1e-3), rand(n, 1e-3).square()) for n in sizes]
    grads = [[rand(n, 1e-3).bfloat16() for n in sizes] for _ in range(2)]
    results = []
    for queued in (False, True):
        state = [tuple(x.clone() for x in part) for part in base]
        torch.cuda.synchronize()
        stream = torch.cuda.Stream()
        lc = P.LayerCheck(stream=stream, mode=P.LC_DRIFT_ACCUMULATE, copy_engine=engine)
        lc.register_layout([P.segment(k, w, None, m, v) for k, (w, m, v) in enumerate(state)], len(sizes))
        for t in (1, 2):
            lc.register_optimizer(grads[t - 1])
            if queued and t == 1:
                with torch.cuda.stream(stream):
                    torch.cuda._sleep(1 << 29)       # a quarter of a second or more
            lc.adamw_step_measure(t, lr=1e-3, weight_decay=0.1)
            if not queued:
                torch.cuda.synchronize()
            if t == 1:
                if queued:
                    lc.register_optimizer(grads[1])
                lc.select(1e12, 1 << 30)             # closes the step
        torch.cuda.synchronize()
        results.append([x for part in state for x in part])
        lc.close()
    for a, b in zip(*results):
        assert torch.equal(a.view(torch.int32), b.view(torch.int32))
