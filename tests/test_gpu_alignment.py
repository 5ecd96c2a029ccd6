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


@pytest.mark.parametrize("staging", [0, 2 << 20])
@pytest.mark.parametrize("fuse", [True, False])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_pack_commit_restore_off_alignment(dtype, fuse, staging):
    """Weights, references and moments each at their own offset from a
    16-byte boundary: the packed stream (to the device, or through a store
    with `staging` bytes of ring, whose launches end inside sections), the
    committed references and the restored tensors equal the sources byte for
    byte, padding is zero and nothing beside them is written."""
    torch = require_gpu()
    import paper_2609_27193_gb300 as P
    esz = 2 if dtype == "bf16" else 4
    tt = torch.bfloat16 if dtype == "bf16" else torch.float32
    g = torch.Generator(device="cuda").manual_seed(esz + fuse)
    sizes = [1, 2, 7, 8, 9, 17, 33, 63, 64, 65, 24575, 24576, 24577, 1000003]
    segs, keep = [], []
    for k, n in enumerate(sizes * (16 // esz // 2)):
        offs = (esz * k % 16, esz * (k // 2 + k // len(sizes)) % 16, 4 * k % 16, 4 * (k + k // 3) % 16)
        part = [_placed(torch, n, d, o) + (o,) for d, o in zip((tt, tt, torch.float32, torch.float32), offs)]
        for _, view, _ in part:
            view.copy_(torch.randn(n, generator=g, device="cuda"))
        keep.append(part)
        segs.append(P.segment(k // 3, part[0][1], part[1][1], part[2][1], part[3][1]))
    N = segs[-1].layer + 1
    more = dict(staging_bytes=staging) if staging else {}
    lc = P.LayerCheck(fuse_commit=fuse, **more)
    lc.register_layout(segs, N)
    lc.measure(1)
    mask, _, nbytes = lc.select(1e-3, 0)
    assert mask.all()
    raw = lambda x: x.contiguous().view(torch.uint8)
    want = []
    for l in range(N):
        members = [keep[k] for k, s in enumerate(segs) if s.layer == l]
        for part in (0, 2, 3):
            for m in members:
                b = raw(m[part][1])
                want.append(b)
                want.append(torch.zeros(-b.numel() % 256, dtype=torch.uint8, device="cuda"))
    want = torch.cat(want)
    assert want.numel() == nbytes
    src = [[p[1].clone() for p in part] for part in keep]
    if staging:
        store = P.Store(lc, capacity_bytes=nbytes + (1 << 20))
        lc.pack_async(store)
    else:
        dst = torch.full((nbytes + 64,), 0xA5, dtype=torch.uint8, device="cuda")
        lc.pack_device(dst)
    lc.commit_snapshot()
    if staging:
        lc.wait_durable(1)
        got = np.concatenate([store.block(i) for i in range(len(store))])
        assert np.array_equal(got, want.cpu().numpy())
    else:
        torch.cuda.synchronize()
        assert torch.equal(dst[:nbytes], want) and set(dst[nbytes:].tolist()) == {0xA5}
    for part, old in zip(keep, src):
        assert torch.equal(raw(part[1][1]), raw(old[0])), "reference"
        if staging:
            for x in part:
                x[1].zero_()
    if staging:
        torch.cuda.synchronize()
        lc.restore(store, 1)
        for part, old in zip(keep, src):
            for j, k in ((0, 0), (1, 0), (2, 2), (3, 3)):
                assert torch.equal(raw(part[j][1]), raw(old[k])), "restored"
    for part in keep:
        for buf, view, o in part:
            assert set(_outside(buf, view, o)) == {0xA5}, "bytes beside a tensor were written"
    lc.close()


@pytest.mark.parametrize("grad_dtype", ["bf16", "f32"])
@pytest.mark.parametrize("lead", [0, 8])
def test_adamw_off_alignment(lead, grad_dtype):
    """The fused step with moments, gradients and model copies at every
    offset from the weights' vectors: each array equals the step's fp32
    operations done one by one on the CPU, bit for bit, and nothing beside
    it is written.  The sums are within the roundings of a chunk's chains
    (three terms and a tree of four) of the 64-bit ones."""
    torch = require_gpu()
    import paper_2609_27193_gb300 as P
    gt = torch.bfloat16 if grad_dtype == "bf16" else torch.float32
    gsz = 2 if grad_dtype == "bf16" else 4
    g = torch.Generator().manual_seed(lead + gsz)
    hp = dict(lr=1e-3, beta1=0.9, beta2=0.95, eps=1e-8, weight_decay=0.1)
    sizes = [1, 2, 3, 4, 5, 8, 9, 11, 31, 257, 2047, 2048, 2049, 4100, 100003]
    combos = [(4 * (k % 4), 4 * (k // 4 % 4), gsz * (k % (16 // gsz)), 2 * ((3 * k + 1) % 8)) for k in range(16)]
    segs, keep, grads, models = [], [], [], []
    for k, (om, ov, og, oc) in enumerate(combos):
        for n in sizes:
            p = torch.randn(n, generator=g) * 0.02
            m = torch.randn(n, generator=g) * 1e-3
            v = torch.randn(n, generator=g).abs() * 1e-6
            x = (torch.randn(n, generator=g) * 1e-3).to(gt)
            part = [_placed(torch, n, d, o) + (o,) for d, o in
                    ((torch.float32, lead), (torch.float32, om), (torch.float32, ov), (gt, og), (torch.bfloat16, oc))]
            for t, src in zip(part, (p, m, v, x)):
                t[1].copy_(src)
            keep.append((part, p, m, v, x))
            segs.append(P.segment(k, part[0][1], None, part[1][1], part[2][1]))
            grads.append(part[3][1])
            models.append(part[4][1])
    N = len(combos)
    lc = P.LayerCheck(mode=P.LC_DRIFT_ACCUMULATE)
    lc.register_layout(segs, N)
    lc.register_optimizer(grads, models)
    sums = torch.zeros(3 * N, dtype=torch.float64, device="cuda")
    lc.set_layer_sums_buffer(sums)
    lc.adamw_step_measure(1, **hp)
    torch.cuda.synchronize()
    f = lambda x: torch.tensor(np.float32(x))
    want = np.zeros((N, 3))
    for s, (part, p, m, v, x) in zip(segs, keep):
        x = x.float()
        m2 = m * f(0.9) + x * f(1 - 0.9)
        v2 = v * f(0.95) + (x * x) * f(1 - 0.95)
        vh = v2 * f(1 / (1 - 0.95))
        p2 = p * f(1 - 1e-3 * 0.1) - (m2 * f(1e-3 / (1 - 0.9))) / (torch.sqrt(vh) + f(1e-8))
        want[s.layer] += ((p2 - p).abs().double().sum().item(), p.abs().double().sum().item(), p.numel())
        for t, ref in zip((part[0], part[1], part[2]), (p2, m2, v2)):
            assert torch.equal(t[1].cpu().view(torch.int32), ref.view(torch.int32)), (s.layer, p.numel())
        assert torch.equal(part[4][1].cpu().view(torch.int16), p2.to(torch.bfloat16).view(torch.int16))
        for buf, view, o in part:
            assert set(_outside(buf, view, o)) == {0xA5}, "bytes beside an array were written"
    got = sums.cpu().numpy().reshape(N, 3)
    assert np.array_equal(got[:, 2], want[:, 2])
    assert (np.abs(got - want) <= 5 * 2.0 ** -24 * np.abs(want)).all()
    assert lc.counters()["bulk_measure_launches"] == 1
    lc.close()


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_noalloc_measure_off_alignment(dtype):
    """lc_measure_noalloc over references at every offset from the weights,
    sizes at the ends of vectors and chunks, layers in shuffled order: exact
    sums, and again on the next call with other values."""
    torch = require_gpu()
    import ctypes as C
    import paper_2609_27193_gb300 as P
    from paper_2609_27193_gb300 import _abi
    esz = 2 if dtype == "bf16" else 4
    tt = torch.bfloat16 if dtype == "bf16" else torch.float32
    g = torch.Generator(device="cuda").manual_seed(esz)
    keep = []
    for n in SIZES:
        for shift in range(0, 16, esz):
            lead = esz * (len(keep) % (16 // esz))
            keep.append((_placed(torch, n, tt, lead)[1], _placed(torch, n, tt, (lead + shift) % 16)[1]))
    N = len(keep)
    order = np.random.default_rng(esz).permutation(N)
    segs = (_abi.lc_segment * N)(*[P.segment(int(k), *keep[k]) for k in order])
    out = torch.empty(3 * N, dtype=torch.float64, device="cuda")
    for _ in range(2):
        for w, r in keep:
            w.copy_(_grid(torch, w.numel(), g))
            r.copy_(_grid(torch, w.numel(), g))
        out.fill_(float("nan"))
        _abi.check(P.library().lc_measure_noalloc(0, C.c_void_p(torch.cuda.current_stream().cuda_stream), segs, N, N,
                                                  C.c_void_p(out.data_ptr())))
        got = out.cpu().numpy().reshape(N, 3)
        for k, (w, r) in enumerate(keep):
            d, a = (w.double() - r.double()).abs().sum().item(), r.double().abs().sum().item()
            assert got[k].tolist() == [d, a, w.numel()], (k, w.numel())
