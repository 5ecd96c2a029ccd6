"""Library calls inside a caller's CUDA graph: the allocation-free measure
and lc_measure only launch kernels, so a capture holds them and every replay
measures the tensors as they are then."""
import ctypes as C

import numpy as np
import pytest

from tests.lc_harness import require_gpu

pytestmark = pytest.mark.gpu

UNIT = 2.0 ** -10


@pytest.mark.parametrize("call", ["noalloc", "measure"])
def test_measures_in_a_callers_graph(call):
    """Small integers on a 2^-10 grid: the sums are exact on every replay."""
    torch = require_gpu()
    import paper_2609_27193_gb300 as P
    from paper_2609_27193_gb300 import _abi
    g = torch.Generator(device="cuda").manual_seed(1)
    w = [torch.zeros(n, dtype=torch.bfloat16, device="cuda") for n in (70001, 4096, 33)]
    r = [torch.zeros_like(x) for x in w]

    def fill():
        for x in w + r:
            x.copy_(torch.randint(-8, 9, (x.numel(),), generator=g, device="cuda").float() * UNIT)

    segs = [P.segment(k, w[k], r[k]) for k in range(3)]
    arr = (_abi.lc_segment * 3)(*segs)
    out = torch.zeros(9, dtype=torch.float64, device="cuda")
    stream = torch.cuda.Stream()
    lc = P.LayerCheck(stream=stream)
    lc.register_layout(segs, 3)
    lc.set_layer_sums_buffer(out)

    def noalloc():
        _abi.check(P.library().lc_measure_noalloc(0, C.c_void_p(torch.cuda.current_stream().cuda_stream), arr, 3, 3,
                                                  C.c_void_p(out.data_ptr())))

    fill()
    torch.cuda.synchronize()
    noalloc()                                  # the device's set-up, before any capture
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        noalloc() if call == "noalloc" else lc.measure(1)
    for _ in range(3):
        fill()
        out.fill_(float("nan"))
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        want = [[(a.double() - b.double()).abs().sum().item(), b.double().abs().sum().item(), a.numel()]
                for a, b in zip(w, r)]
        assert np.array_equal(out.cpu().numpy().reshape(3, 3), want)
    lc.close()
