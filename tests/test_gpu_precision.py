"""What the chains with recovered rounding errors are for: the sums of
tensors off one another's alignment, over values that every addition rounds.
Their terms are fp32, so the reference is the exact sum of those terms
(math.fsum) and only the additions can differ."""
import math

import numpy as np
import pytest

from tests.lc_harness import require_gpu

pytestmark = pytest.mark.gpu

# At most 28 terms in a chain of a chunk: the recovered errors are below
# 28 * 2^-24 of it and lose 28 times 2^-24 of that themselves, 2^-38.4 in all;
# the fp64 additions are far below.  Plain fp32 chains are off by 2^-30 and more.
RTOL = 2.0 ** -38

SIZES = [5, 250, 6000, 12289, 70001, 400009]


def _at(torch, n, dtype, offset):
    size = torch.empty(0, dtype=dtype).element_size() * n
    return torch.zeros(16 + size + 16, dtype=torch.uint8, device="cuda")[offset:offset + size].view(dtype)


def _values(torch, spread, n, g):
    """Normal values, or such values over 30 binades."""
    x = torch.randn(n, generator=g, device="cuda") * 0.02
    if spread == "wide":
        x *= torch.exp2(torch.rand(n, generator=g, device="cuda") * 30 - 15)
    return x


def _exact(terms):
    return math.fsum(terms.double().cpu().numpy().tolist())


@pytest.mark.parametrize("call", ["snapshot", "accumulate", "noalloc"])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("spread", ["normal", "wide"])
def test_sums_off_alignment_keep_their_precision(spread, dtype, call):
    """Layers of one tensor each, R at every offset but W's own."""
    torch = require_gpu()
    import ctypes as C
    import paper_2609_27193_gb300 as P
    from paper_2609_27193_gb300 import _abi
    esz = 2 if dtype == "bf16" else 4
    tt = torch.bfloat16 if dtype == "bf16" else torch.float32
    g = torch.Generator(device="cuda").manual_seed(esz)
    segs, want = [], []
    for n in SIZES:
        for shift in range(esz, 16, esz):
            lead = esz * (len(segs) % (16 // esz))
            w, r = _at(torch, n, tt, lead), _at(torch, n, tt, (lead + shift) % 16)
            r.copy_(_values(torch, spread, n, g))
            w.copy_(_values(torch, spread, n, g) if len(segs) % 2 else
                    r.float() * (1 + 0.01 * torch.randn(n, generator=g, device="cuda")))
            want.append((_exact((w.float() - r.float()).abs()), _exact(r.float().abs()), n))
            segs.append(P.segment(len(segs), w, r))
    N = len(segs)
    sums = torch.zeros(3 * N, dtype=torch.float64, device="cuda")
    if call == "noalloc":
        _abi.check(P.library().lc_measure_noalloc(0, C.c_void_p(torch.cuda.current_stream().cuda_stream),
                                                  (_abi.lc_segment * N)(*segs), N, N, C.c_void_p(sums.data_ptr())))
    else:
        lc = P.LayerCheck(mode=P.LC_DRIFT_ACCUMULATE if call == "accumulate" else P.LC_DRIFT_SNAPSHOT)
        lc.register_layout(segs, N)
        lc.set_layer_sums_buffer(sums)
        lc.measure(1)
    torch.cuda.synchronize()
    got, want = sums.cpu().numpy().reshape(N, 3), np.array(want)
    assert np.array_equal(got[:, 2], want[:, 2])
    assert (np.abs(got - want) <= RTOL * np.abs(want)).all(), np.abs(got / want - 1).max(axis=0)


@pytest.mark.parametrize("form", ["gradients", "moments"])
@pytest.mark.parametrize("grad_dtype", ["bf16", "f32"])
@pytest.mark.parametrize("spread", ["normal", "wide"])
def test_fused_step_sums_off_alignment_keep_their_precision(spread, grad_dtype, form):
    """Gradients, or moments and gradients, off the weights' alignment: sums
    of the update as it was stored."""
    torch = require_gpu()
    import paper_2609_27193_gb300 as P
    gt = torch.bfloat16 if grad_dtype == "bf16" else torch.float32
    gsz = 2 if grad_dtype == "bf16" else 4
    g = torch.Generator(device="cuda").manual_seed(gsz)
    segs, grads, old = [], [], []
    for k, n in enumerate(SIZES):
        at = 4 * (k % 3 + 1) if form == "moments" else 0
        w, m, v = (_at(torch, n, torch.float32, o) for o in (0, at, at))
        x = _at(torch, n, gt, gsz)
        w.copy_(_values(torch, spread, n, g))
        x.copy_(torch.randn(n, generator=g, device="cuda") * 1e-3)
        v.copy_(torch.rand(n, generator=g, device="cuda") * 1e-6)
        old.append(w.clone())
        segs.append(P.segment(k, w, None, m, v))
        grads.append(x)
    N = len(segs)
    lc = P.LayerCheck(mode=P.LC_DRIFT_ACCUMULATE)
    lc.register_layout(segs, N)
    lc.register_optimizer(grads)
    sums = torch.zeros(3 * N, dtype=torch.float64, device="cuda")
    lc.set_layer_sums_buffer(sums)
    lc.adamw_step_measure(1, lr=1e-3, weight_decay=0.1)
    torch.cuda.synchronize()
    got = sums.cpu().numpy().reshape(N, 3)
    want = np.array([(_exact((s._refs[0] - p).abs()), _exact(p.abs()), p.numel()) for s, p in zip(segs, old)])
    assert np.array_equal(got[:, 2], want[:, 2])
    assert (np.abs(got - want) <= RTOL * np.abs(want)).all(), np.abs(got / want - 1).max(axis=0)


def test_large_layout_off_alignment():
    """A layout whose shifted runs are shared from the larger pool: one layer
    of small integers on a 2^-10 grid, exact in fp32 chunk by chunk."""
    torch = require_gpu()
    import paper_2609_27193_gb300 as P
    g = torch.Generator(device="cuda").manual_seed(7)
    n = 50000003
    segs, want = [], np.zeros((2, 3))
    for k in range(3):
        w, r = _at(torch, n, torch.bfloat16, 2 * k), _at(torch, n, torch.bfloat16, 10)
        for x in (w, r):
            x.copy_(torch.randint(-8, 9, (n,), generator=g, device="cuda", dtype=torch.int8).bfloat16() * 2.0 ** -10)
        d = (w - r).abs().sum(dtype=torch.float64).item()
        want[k // 2] += (d, r.abs().sum(dtype=torch.float64).item(), n)
        segs.append(P.segment(k // 2, w, r))
    lc = P.LayerCheck()
    lc.register_layout(segs, 2)
    sums = torch.zeros(6, dtype=torch.float64, device="cuda")
    lc.set_layer_sums_buffer(sums)
    lc.measure(1)
    torch.cuda.synchronize()
    assert sums.cpu().numpy().reshape(2, 3).tolist() == want.tolist()
    assert lc.counters()["measure_pool_units"] > 0
    lc.close()


EXTREMES = [("large", 2.0 ** 126), ("inf", float("inf")), ("nan", float("nan"))]


@pytest.mark.parametrize("what,value", EXTREMES)
@pytest.mark.parametrize("call", ["snapshot", "accumulate", "noalloc"])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_extreme_values_off_alignment(dtype, call, what, value):
    """Weights, and references, near the end of fp32's range, infinite or NaN
    in runs off one another's alignment, beside a run of ordinary ones: the
    sums are what fp64 addition of the fp32 terms gives."""
    torch = require_gpu()
    import ctypes as C
    import paper_2609_27193_gb300 as P
    from paper_2609_27193_gb300 import _abi
    n = 20000
    tt = torch.bfloat16 if dtype == "bf16" else torch.float32
    pairs = [(_at(torch, n, tt, 4), _at(torch, n, tt, 12)) for _ in range(3)]
    for x in (pairs[0][0], pairs[1][1]):
        if what == "large":
            x.fill_(value)
        else:
            x[n // 2] = value
    pairs[2][0].fill_(0.5)
    pairs[2][1].fill_(0.25)
    segs = [P.segment(k, w, r) for k, (w, r) in enumerate(pairs)]
    sums = torch.zeros(9, dtype=torch.float64, device="cuda")
    if call == "noalloc":
        _abi.check(P.library().lc_measure_noalloc(0, C.c_void_p(torch.cuda.current_stream().cuda_stream),
                                                  (_abi.lc_segment * 3)(*segs), 3, 3, C.c_void_p(sums.data_ptr())))
    else:
        lc = P.LayerCheck(mode=P.LC_DRIFT_ACCUMULATE if call == "accumulate" else P.LC_DRIFT_SNAPSHOT)
        lc.register_layout(segs, 3)
        lc.set_layer_sums_buffer(sums)
        lc.measure(1)
    torch.cuda.synchronize()
    x = n * value if what == "large" else value
    want = [[x, 0.0, n], [x, x, n], [n * 0.25, n * 0.25, n]]
    assert np.array_equal(sums.cpu().numpy().reshape(3, 3), want, equal_nan=True)
    if call == "accumulate":
        for w, r in pairs:
            assert torch.equal(w.view(torch.uint8), r.view(torch.uint8))


@pytest.mark.parametrize("what,value", EXTREMES)
@pytest.mark.parametrize("form", ["gradients", "moments"])
def test_fused_step_extreme_values_off_alignment(form, what, value):
    """The same for the fused step's loose forms: no gradient, a decay that
    halves every weight (an infinite one stays, so its update is NaN)."""
    torch = require_gpu()
    import paper_2609_27193_gb300 as P
    n, at = 20000, 8 if form == "moments" else 0
    segs, grads, ws = [], [], []
    for k in range(2):
        w, m, v, x = (_at(torch, n, torch.float32, o) for o in (0, at, at, 4))
        if k == 1:
            w.fill_(0.5)
        elif what == "large":
            w.fill_(value)
        else:
            w[n // 2] = value
        segs.append(P.segment(k, w, None, m, v))
        grads.append(x)
        ws.append(w)
    lc = P.LayerCheck(mode=P.LC_DRIFT_ACCUMULATE)
    lc.register_layout(segs, 2)
    lc.register_optimizer(grads)
    sums = torch.zeros(6, dtype=torch.float64, device="cuda")
    lc.set_layer_sums_buffer(sums)
    lc.adamw_step_measure(1, lr=1.0, weight_decay=0.5)
    torch.cuda.synchronize()
    d, a = (n * value / 2, n * value) if what == "large" else (float("nan"), value)
    assert np.array_equal(sums.cpu().numpy().reshape(2, 3), [[d, a, n], [n * 0.25, n * 0.5, n]], equal_nan=True)
    assert (ws[1] == 0.25).all()
