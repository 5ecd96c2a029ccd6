"""Tensors that do not start on 16-byte boundaries: weights, references,
moments and gradients at every offset that their element sizes allow, in the
sizes where a vector, a chunk or a work range ends.  Values sit on a 2^-10
grid of small integers, so every sum is exact in fp32 and the comparison is
for equality."""
import numpy as np
import pytest

from tests.lc_harness import require_gpu

pytestmark = pytest.mark.gpu

UNIT = 2.0 ** -10
GUARD = 64            # bytes of a known pattern on both sides of every tensor


def _placed(torch, n, dtype, offset, fill=0xA5):
    """(buffer, view): n elements `offset` bytes past a 256-byte boundary,
    the rest of the buffer filled with a pattern."""
    size = torch.empty(0, dtype=dtype).element_size() * n
    buf = torch.full((GUARD + 16 + size + GUARD,), fill, dtype=torch.uint8, device="cuda")
    return buf, buf[GUARD + offset:GUARD + offset + size].view(dtype)


def _outside(buf, view, offset):
    size = view.numel() * view.element_size()
    return buf[:GUARD + offset].tolist() + buf[GUARD + offset + size:].tolist()


def _grid(torch, n, g):
    return torch.randint(-8, 9, (n,), generator=g, device="cuda").float() * UNIT


SIZES = [1, 2, 7, 8, 9, 15, 16, 17, 24, 25, 33, 257, 12287, 12288, 12289, 24576 + 5, 100003]


@pytest.mark.parametrize("engine", ["bulk", "threads"])
@pytest.mark.parametrize("mode", ["snapshot", "accumulate"])
@pytest.mark.parametrize("dtype,lead", [("bf16", 0), ("bf16", 6), ("bf16", 14), ("f32", 0), ("f32", 8)])
def test_measure_of_references_off_the_weights_alignment(dtype, lead, mode, engine):
    """W `lead` bytes and R any other offset past a 16-byte boundary: D, A
    and n of every layer (one tensor each) are exact; in accumulate mode R
    equals W afterwards and nothing beside R is written."""
    torch = require_gpu()
    import paper_2609_27193_gb300 as P
    esz = 2 if dtype == "bf16" else 4
    tt = torch.bfloat16 if dtype == "bf16" else torch.float32
    g = torch.Generator(device="cuda").manual_seed(lead + esz)
    segs, keep = [], []
    for n in SIZES:
        for shift in range(0, 16, esz):
            wb, w = _placed(torch, n, tt, lead)
            ro = (lead + shift) % 16
            rb, r = _placed(torch, n, tt, ro)
            w.copy_(_grid(torch, n, g))
            r.copy_(_grid(torch, n, g))
            keep.append((w, rb, r, ro, r.clone()))
            segs.append(P.segment(len(segs), w, r))
    N = len(segs)
    lc = P.LayerCheck(copy_engine=engine, mode=P.LC_DRIFT_ACCUMULATE if mode == "accumulate" else P.LC_DRIFT_SNAPSHOT)
    lc.register_layout(segs, N)
    sums = torch.zeros(3 * N, dtype=torch.float64, device="cuda")
    lc.set_layer_sums_buffer(sums)
    lc.measure(1)
    torch.cuda.synchronize()
    got = sums.cpu().numpy().reshape(N, 3)
    for k, (w, rb, r, ro, old) in enumerate(keep):
        d = float((w.double() - old.double()).abs().sum())
        a = float(old.double().abs().sum())
        assert got[k].tolist() == [d, a, w.numel()], (k, w.numel(), ro)
        if mode == "accumulate":
            assert torch.equal(r, w), (w.numel(), ro)
        assert set(_outside(rb, r, ro)) == {0xA5}, "bytes beside R were written"
    assert lc.counters()["bulk_measure_launches"] == (1 if engine == "bulk" else 0)
    lc.close()


@pytest.mark.parametrize("what,value", [("large", 2.0 ** 126), ("inf", float("inf")), ("nan", float("nan"))])
def test_measure_of_extreme_values_off_alignment(what, value):
    """Weights near the end of fp32's range, infinite and NaN ones, in runs
    whose references lie elsewhere: the sums are what fp64 addition gives."""
    torch = require_gpu()
    import paper_2609_27193_gb300 as P
    n = 20000
    keep = [_placed(torch, n, torch.float32, 4) + _placed(torch, n, torch.float32, 12) for _ in range(2)]
    (_, w, _, r), (_, w1, _, r1) = keep
    w.fill_(value) if what == "large" else w.zero_()
    r.zero_()
    if what != "large":
        w[n // 2] = value
    w1.fill_(0.5)
    r1.fill_(0.25)
    lc = P.LayerCheck()
    lc.register_layout([P.segment(0, w, r), P.segment(1, w1, r1)], 2)
    sums = torch.zeros(6, dtype=torch.float64, device="cuda")
    lc.set_layer_sums_buffer(sums)
    lc.measure(1)
    torch.cuda.synchronize()
    got = sums.cpu().numpy().reshape(2, 3)
    want = n * value if what == "large" else value
    assert np.array_equal(got[0], [want, 0.0, n], equal_nan=True)
    assert got[1].tolist() == [n * 0.25, n * 0.25, n]
    lc.close()
