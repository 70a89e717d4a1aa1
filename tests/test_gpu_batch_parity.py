"""The persistent batch schedule where every order's staging barriers are used again and again.

A CTA keeps a set of barriers for each order and runs through their phases tile by tile; at p = 3 a warp
has barriers of its own.  The batch gives every order more than twice as many volume tiles as the launch
has CTAs (three per SM: 168 registers a thread leave no room for a fourth), so that at each order CTAs go
through both parities.  Same tolerance as the small batch's: 1e-6 of the state's scale against the orders
one after another, and no wait that ran out.
"""
import collections

import numpy as np
import pytest

from chorus_inputs import BatchConfig, make_phys

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TILE = {2: 14, 3: 8, 4: 5, 5: 3}  # elements per CTA of the persistent launch


def test_every_order_reuses_its_barriers():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1503_00834_gb300 import ChorusError, Shells, build

    build.build()
    cfg = BatchConfig("batch_parity", 12, 11, 9, 14, 4, 8, (2, 3, 4, 5), 0.75, 1.0, 1e-3,
                      make_phys(0.75, 1.5, 3.0, 1e-3))
    elems = collections.Counter()
    for s in cfg.shells():
        elems[s.p] += 6 * s.n * s.n * s.n_r
    ctas = 3 * torch.cuda.get_device_properties(0).multi_processor_count
    for p, epb in TILE.items():
        assert -(-elems[p] // epb) > 2 * ctas, (p, elems[p])
    sh = Shells(cfg)
    b = sh.batch
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
