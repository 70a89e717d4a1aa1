"""Calls after a staging wait that ran out, while nobody has read the error flag yet.

A wait that gives up costs its own elements, which keep their old contents, and sets the flag that
chorus_check reports once; it must not hold up later work on the mesh.  With the wait limit at zero every
element of a call is left alone; the next calls, with the default limit and the flag still set, have to
be complete: bit for bit the results of a mesh that never timed out.  Both forms, at an order whose
elements are staged by warps (p = 3) and one that stages by CTA (p = 4).
"""
import ctypes

import pytest

from chorus_inputs import small_shell

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ETIMEOUT = 6


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1503_00834_gb300 import build

    build.build()


@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "fp32"])
@pytest.mark.parametrize("p", [3, 4])
def test_later_calls_are_complete_with_the_flag_unread(p, prec):
    from paper_1503_00834_gb300 import ChorusError, Shell, native

    cfg = small_shell(3, 2, p)
    sh = Shell(cfg)
    m = sh.mesh
    dtype = torch.float64 if prec == 0 else torch.float32
    q0 = torch.empty(m.state_shape(), dtype=dtype, device="cuda")
    m.state_init(sh.params, cfg.seed, cfg.entropy_amp, prec, q0)
    ws = torch.empty(m.workspace_bytes(prec), dtype=torch.uint8, device="cuda")
    calls = {
        "residual": lambda q, R: m.residual(sh.params, prec, q, R, ws),
        "noalloc": lambda q, R: native._ok("noalloc", native.load().chorus_residual_noalloc(
            m.handle, ctypes.byref(sh.params), prec, native._ptr(q), native._ptr(R), native._stream(None))),
        "rk3": lambda q, R: m.rk_step(sh.params, prec, q, ws, sh.dt, 2),
        "rk54": lambda q, R: m.rk_step_scheme(sh.params, prec, 1, q, ws, sh.dt, 1),
    }

    def run(name):
        q, R = q0.clone(), torch.full_like(q0, 12345.0)
        calls[name](q, R)
        return q, R

    want = {name: run(name) for name in calls}
    m.check()
    try:
        m.set_wait_limit(0)
        for name in calls:
            q, R = run(name)
            assert torch.equal(q, q0) and bool(torch.all(R == 12345.0)), name
        m.set_wait_limit(-1)
        for name in calls:  # the flag is still set
            q, R = run(name)
            assert torch.equal(q, want[name][0]) and torch.equal(R, want[name][1]), name
    finally:
        m.set_wait_limit(-1)
    with pytest.raises(ChorusError) as e:
        m.check()
    assert e.value.status == ETIMEOUT
    m.check()
    for name in calls:
        q, R = run(name)
        assert torch.equal(q, want[name][0]) and torch.equal(R, want[name][1]), name
