"""A decision whose call ran out of time, asked for again."""
import numpy as np
import pytest

from oracle import oracle as O
from tests.lc_harness import require_gpu

pytestmark = pytest.mark.gpu

BUSY = 1 << 29        # cycles (a quarter of a second or more) that the stream is kept busy


@pytest.mark.parametrize("again", ["same", "other"])
@pytest.mark.parametrize("mode", ["snapshot", "accumulate"])
def test_select_repeated_after_a_timeout(mode, again):
    """lc_select gives up while the stream is busy with other work and its
    kernel is still to come: the repeated call (with the same thresholds or
    with others) decides as if it were the only one, over two attempts that
    run out of time, and the following steps find the state that it left.
    u injected per layer (D = u, A = 0, n = 1 with eps_w = 1)."""
    torch = require_gpu()
    import paper_2609_27193_gb300 as P
    omode = O.SNAPSHOT if mode == "snapshot" else O.ACCUMULATE
    N = 40
    w = [torch.zeros(16, device="cuda") for _ in range(N)]
    r = [torch.zeros(16, device="cuda") for _ in range(N)]
    lc = P.LayerCheck(eps_w=1.0, timeout_ms=20,
                      mode=P.LC_DRIFT_SNAPSHOT if mode == "snapshot" else P.LC_DRIFT_ACCUMULATE)
    lc.register_layout([P.segment(k, w[k], r[k]) for k in range(N)], N)
    sums = torch.zeros(3 * N, dtype=torch.float64, device="cuda")
    lc.set_layer_sums_buffer(sums)
    rng = np.random.default_rng(5)
    delta, tl = np.zeros(N), np.zeros(N, dtype=np.int64)
    tau, k = 0.5, 3
    for t in range(1, 9):
        lc.measure(t)
        us = rng.choice([0.0, tau / 4, tau / 2, tau], N)
        inj = np.zeros((N, 3))
        inj[:, 0], inj[:, 2] = us, 1.0
        sums.copy_(torch.from_numpy(inj.reshape(-1)))
        late = t in (2, 5, 6)
        for _ in range(2 if late else 0):
            torch.cuda._sleep(BUSY)
            with pytest.raises(P.LCError) as e:
                lc.select(tau / 2 if again == "other" else tau, 1 if again == "other" else k)
            assert e.value.status == 6                     # LC_ERR_TIMEOUT
        if late:
            torch.cuda.synchronize()
        mask, u, _ = lc.select(tau, k)
        omask, _, _ = O.select_step(us, delta, tl, tau, k, t, omode)
        assert mask.tolist() == omask.tolist(), t
        assert u.tolist() == us.tolist()
        info = lc.info()
        mx, wt = O.staleness(tl, np.full(N, 16), t)
        assert info["max_staleness"] == mx and info["weighted_staleness"] == wt
        dst = torch.empty(max(16, info["bytes"]), dtype=torch.uint8, device="cuda")
        lc.pack_device(dst)
        lc.commit_snapshot()
        torch.cuda.synchronize()
    lc.close()
