"""The measure's combine over numbers of layers around its tile of 512: the
sums themselves, of every kernel that has a combine."""
import numpy as np
import pytest

from tests.lc_harness import require_gpu

pytestmark = pytest.mark.gpu

UNIT = 2.0 ** -10


@pytest.mark.parametrize("call", ["snapshot", "accumulate", "threads", "adamw"])
@pytest.mark.parametrize("nlayers", [1, 511, 512, 513, 1024, 1025, 2500])
def test_sums_of_many_layers(nlayers, call):
    """Layers of one to three tensors of up to 3000 elements, one of them a
    hundred times as large; small integers on a 2^-10 grid, so that sums are
    exact.  The fused step moves every weight by a whole unit (moments and
    gradients zero, weight decay 1, learning rate 1: w becomes 0)."""
    torch = require_gpu()
    import paper_2609_27193_gb300 as P
    fused = call == "adamw"
    rng = np.random.default_rng(nlayers)
    tt = torch.float32 if fused else torch.bfloat16
    layer = np.repeat(np.arange(nlayers), rng.integers(1, 4, nlayers))
    numel = rng.integers(1, 3000, layer.size)
    numel[layer.size // 2] = 300000
    off = np.concatenate([[0], np.cumsum(numel)])
    g = torch.Generator(device="cuda").manual_seed(nlayers)
    grid = lambda: (torch.randint(-8, 9, (int(off[-1]),), generator=g, device="cuda").float() * UNIT).to(tt)
    w, r = grid(), grid()
    zero = [torch.zeros(int(off[-1]), device="cuda") for _ in range(3)] if fused else None
    cut = lambda x, k: x[off[k]:off[k + 1]]
    segs = [P.segment(int(layer[k]), cut(w, k), None if fused else cut(r, k),
                      *((cut(zero[0], k), cut(zero[1], k)) if fused else ())) for k in range(layer.size)]
    a = (w if fused else r).double().abs()
    d = a if fused else (w.double() - r.double()).abs()
    per = lambda x: np.add.reduceat(x.cpu().numpy(), off[:-1])
    want = np.zeros((nlayers, 3))
    for c, x in enumerate((per(d), per(a), numel)):
        np.add.at(want[:, c], layer, x)
    lc = P.LayerCheck(mode=P.LC_DRIFT_SNAPSHOT if call in ("snapshot", "threads") else P.LC_DRIFT_ACCUMULATE,
                      copy_engine="threads" if call == "threads" else "bulk")
    lc.register_layout(segs, nlayers)
    sums = torch.full((3 * nlayers,), float("nan"), dtype=torch.float64, device="cuda")
    lc.set_layer_sums_buffer(sums)
    if fused:
        lc.register_optimizer([cut(zero[2], k) for k in range(layer.size)])
        lc.adamw_step_measure(1, lr=1.0, weight_decay=1.0)
    else:
        lc.measure(1)
    torch.cuda.synchronize()
    assert np.array_equal(sums.cpu().numpy().reshape(nlayers, 3), want)
    lc.close()
