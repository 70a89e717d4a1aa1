"""The persistent batch schedule with many work items a CTA, of every order in turn.

A CTA keeps its staging barriers from item to item; the orders use different numbers of them.  The
batch has more tiles of each order than the device holds CTAs, so every CTA takes items of several
orders.  Same tolerance as the small batch's: 1e-6 of the state's scale against the orders one after
another, and no wait that ran out.
"""
import numpy as np
import pytest

from chorus_inputs import BatchConfig, make_phys

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_many_items_of_mixed_orders_per_cta():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1503_00834_gb300 import ChorusError, Shells, build

    build.build()
    cfg = BatchConfig("batch_items", 12, 5, 9, 12, 4, 6, (2, 3, 4, 5), 0.75, 1.0, 1e-3,
                      make_phys(0.75, 1.5, 3.0, 1e-3))
    sh = Shells(cfg)
    b = sh.batch
    assert sorted(set(b.orders)) == [2, 3, 4, 5]
    out = []
    for mode in (b.SERIAL, b.PERSISTENT):
        try:
            b.schedule(mode)
        except ChorusError as e:
            if e.status == 7:  # CHORUS_EUNSUPPORTED
                pytest.skip("no cooperative launch on this device")
            raise
        Q = torch.empty(b.n_state, dtype=torch.float32, device="cuda")
        ws = torch.empty(b.workspace_bytes, dtype=torch.uint8, device="cuda")
        b.init(Q)
        b.rk_step(Q, ws, sh.dt, 3)
        assert np.all(np.isfinite(b.reduce(Q)))  # also reports a wait that ran out
        out.append(Q)
    for s in range(len(sh.cfgs)):
        q, p = b.view(out[0], s), b.view(out[1], s)
        d, scale = (q - p).abs().max().item(), q.abs().max().item()
        assert d <= 1e-6 * scale, (s, sh.cfgs[s].p, d, scale)
