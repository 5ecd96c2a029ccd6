"""lc_measure_noalloc when a wait of its kernel runs out, and over managed
memory, which the bulk engine is not given."""
import ctypes as C

import numpy as np
import pytest

from tests.lc_harness import require_gpu

pytestmark = pytest.mark.gpu

UNIT = 2.0 ** -10


def _grid(torch, n, g):
    return torch.randint(-8, 9, (n,), generator=g, device="cuda").float() * UNIT


def test_a_wait_that_runs_out_leaves_nan_and_the_next_call_is_right():
    """Each CTA's first load announces 16 bytes more than it brings; its wait
    gives up after a second and every value is NaN, element counts too."""
    torch = require_gpu()
    import paper_2609_27193_gb300 as P
    from paper_2609_27193_gb300 import _abi
    lib, g = P.library(), torch.Generator(device="cuda").manual_seed(2)
    sizes = [500000, 33, 70001]
    w = [_grid(torch, n, g).bfloat16() for n in sizes]
    r = [_grid(torch, n, g).bfloat16() for n in sizes]
    segs = (_abi.lc_segment * 3)(*[P.segment(k, w[k], r[k]) for k in range(3)])
    out = torch.zeros(9, dtype=torch.float64, device="cuda")
    stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    call = lambda flags: lib.lc_measure_noalloc_debug(0, stream, segs, 3, 3, C.c_void_p(out.data_ptr()), flags)
    want = np.array([[(a.double() - b.double()).abs().sum().item(), b.double().abs().sum().item(), a.numel()]
                     for a, b in zip(w, r)])
    for flags in (0, _abi.LC_DEBUG_MEASURE_STALL, 0):
        out.zero_()
        _abi.check(call(flags))
        got = out.cpu().numpy().reshape(3, 3)
        assert np.isnan(got).all() if flags else np.array_equal(got, want)
    assert call(4) == _abi.LC_ERR_INVALID_ARG and call(_abi.LC_DEBUG_BULK_STALL) == _abi.LC_ERR_INVALID_ARG


@pytest.mark.parametrize("managed", ["w", "r", "both"])
@pytest.mark.parametrize("shift", [0, 6])
def test_managed_memory(shift, managed):
    """W, R or both in managed memory, beside a layer of device memory, with
    and without a shift between W and R: exact sums, from a context (which
    says that it took no bulk launch) and without one."""
    torch = require_gpu()
    import paper_2609_27193_gb300 as P
    from paper_2609_27193_gb300 import _abi
    for name in ("libcudart.so.13", "libcudart.so", "/usr/local/cuda/lib64/libcudart.so"):
        try:
            rt = C.CDLL(name)
            break
        except OSError:
            rt = None
    if rt is None:
        pytest.skip("no shared CUDA runtime to allocate managed memory with")
    g, n = torch.Generator(device="cuda").manual_seed(4), 70001
    dev = {k: _grid(torch, n, g).bfloat16() for k in ("w", "r", "w1", "r1")}
    at, blocks = {}, []
    try:
        for k, off in (("w", 2), ("r", (2 + shift) % 16)):
            if managed in (k, "both"):
                p = C.c_void_p()
                assert rt.cudaMallocManaged(C.byref(p), C.c_size_t(2 * n + 16), C.c_uint(1)) == 0
                blocks.append(p)
                at[k] = p.value + off
            else:
                blk = torch.empty(2 * n + 16, dtype=torch.uint8, device="cuda")
                dev[k + "_at"] = blk
                at[k] = blk.data_ptr() + off
            torch.cuda.synchronize()
            assert rt.cudaMemcpy(C.c_void_p(at[k]), C.c_void_p(dev[k].data_ptr()), C.c_size_t(2 * n), 4) == 0
        segs = [_abi.lc_segment(0, _abi.LC_BF16, at["w"], at["r"], None, None, n),
                P.segment(1, dev["w1"], dev["r1"])]
        want = [[(dev[a].double() - dev[b].double()).abs().sum().item(), dev[b].double().abs().sum().item(), n]
                for a, b in (("w", "r"), ("w1", "r1"))]
        out = torch.full((6,), float("nan"), dtype=torch.float64, device="cuda")
        _abi.check(P.library().lc_measure_noalloc(0, C.c_void_p(torch.cuda.current_stream().cuda_stream),
                                                  (_abi.lc_segment * 2)(*segs), 2, 2, C.c_void_p(out.data_ptr())))
        assert out.cpu().numpy().reshape(2, 3).tolist() == want
        lc = P.LayerCheck()
        lc.register_layout(segs, 2)
        lc.set_layer_sums_buffer(out)
        out.fill_(float("nan"))
        lc.measure(1)
        torch.cuda.synchronize()
        assert out.cpu().numpy().reshape(2, 3).tolist() == want
        assert lc.counters()["bulk_measure_launches"] == 0
        lc.close()
    finally:
        torch.cuda.synchronize()
        for p in blocks:
            rt.cudaFree(p)
