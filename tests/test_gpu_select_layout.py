"""The select kernel's stream layout and staleness statistics over numbers of
layers around a warp, a tile of layers and several tiles, and over steps
whose weighted staleness leaves the whole numbers that binary64 adds
exactly."""
import numpy as np
import pytest

from oracle import oracle as O
from tests.lc_harness import require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["snapshot", "accumulate"])
@pytest.mark.parametrize("nlayers", [1, 31, 32, 33, 255, 256, 257, 513, 1025])
def test_layout_and_staleness_over_numbers_of_layers(nlayers, mode):
    """u injected per layer (D = u, A = 0, n = 1 with eps_w = 1): masks and
    statistics equal the oracle's, offsets the running block sizes, and the
    packed stream the persisted tensors; the last step is 2^50 later."""
    torch = require_gpu()
    import paper_2609_27193_gb300 as P
    omode = O.SNAPSHOT if mode == "snapshot" else O.ACCUMULATE
    rng = np.random.default_rng(nlayers)
    numel = rng.integers(1, 40, size=nlayers)
    per = rng.integers(1, 4, size=nlayers)                 # tensors of a layer
    flat = torch.arange(int((numel * per).sum()), device="cuda").to(torch.float32)
    snap = torch.zeros_like(flat)
    segs, parts, o = [], [[] for _ in range(nlayers)], 0
    for l in range(nlayers):
        for k in range(per[l]):
            n = int(numel[l])
            parts[l].append(flat[o:o + n])
            segs.append(P.segment(l, flat[o:o + n], snap[o:o + n]))
            o += n
    lc = P.LayerCheck(eps_w=1.0, mode=P.LC_DRIFT_SNAPSHOT if mode == "snapshot" else P.LC_DRIFT_ACCUMULATE)
    lc.register_layout(segs, nlayers)
    sums = torch.zeros(3 * nlayers, dtype=torch.float64, device="cuda")
    lc.set_layer_sums_buffer(sums)
    delta, tl, counts = np.zeros(nlayers), np.zeros(nlayers, dtype=np.int64), numel * per
    tau = 0.5
    for t in (1, 2, 3, 5, 8, 1 << 50):
        lc.measure(t)
        us = rng.choice([0.0, tau / 2, tau, 2 * tau], nlayers)
        if t == 3:
            us[0] = np.nan
        inj = np.zeros((nlayers, 3))
        inj[:, 0], inj[:, 2] = us, 1.0
        sums.copy_(torch.from_numpy(inj.reshape(-1)))
        k = 4 if t < 10 else 1 << 30
        if t > 10:
            us[:] = 0.0
            inj[:, 0] = 0.0
            inj[::3, 0] = 1.0                              # a third persists; the rest is very stale
            us = inj[:, 0]
            sums.copy_(torch.from_numpy(inj.reshape(-1)))
            k = 2 ** 31 - 1
        mask, u, nbytes = lc.select(tau, k)
        omask, _, _ = O.select_step(us, delta, tl, tau, k, t, omode)
        assert mask.tolist() == omask.tolist()
        info = lc.info()
        mx, wt = O.staleness(tl, counts, t)
        assert info["max_staleness"] == mx and info["weighted_staleness"] == wt
        assert info["n_selected"] == int(omask.sum()) and info["n_nonfinite"] == int(np.isnan(us).sum())
        want, off = [], 0
        offsets = lc.offsets()
        for l in np.flatnonzero(omask):
            assert offsets[l] == off
            for x in parts[l]:
                want.append(x.view(torch.uint8))
                want.append(torch.zeros(-x.numel() * 4 % 256, dtype=torch.uint8, device="cuda"))
            off += lc.layer_block_bytes(int(l))
        assert nbytes == off
        if nbytes:
            dst = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
            lc.pack_device(dst)
            assert torch.equal(dst, torch.cat(want))
        lc.commit_snapshot()
    lc.close()
