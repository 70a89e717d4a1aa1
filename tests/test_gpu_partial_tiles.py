"""Both forms and both integrators against the oracle where the last tile is partly filled, every order.

Element counts below one tile and between tiles: the FP64 residual (2, 4 or 6 elements per CTA) within the
backward-error bound of the parity tests, 1e-12 times the oracle residual's own condition number; one
FP32 step of SSP-RK3 and of SSP-RK(5,4), whose stages run on different kernels, within 1e-5 relative on
q' = Q - Q0.
"""
import numpy as np
import pytest

from chorus_inputs import small_shell
from gpu_common import OracleShell, rel_err, to5
from test_gpu_parity import _condition
from test_gpu_volume import SHAPES

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("p", [2, 3, 4, 5])
@pytest.mark.parametrize("n, n_r, N_rho", SHAPES)
def test_residual_and_steps_match_oracle(p, n, n_r, N_rho):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import rk
    from oracle.residual import residual
    from paper_1503_00834_gb300 import FP32_PERT, FP64, Shell, build

    build.build()
    cfg = small_shell(n, n_r, p, N_rho=N_rho)
    sh = Shell(cfg)
    m = sh.mesh
    osh = OracleShell(cfg)
    W = osh.weights()
    Q = osh.initial_state()

    def state(prec, dtype):
        q = torch.empty(m.state_shape(), dtype=dtype, device="cuda")
        m.state_init(sh.params, cfg.seed, cfg.entropy_amp, prec, q)
        return q, torch.empty(m.workspace_bytes(prec), dtype=torch.uint8, device="cuda")

    q, ws = state(FP64, torch.float64)
    R = torch.empty_like(q)
    m.residual(sh.params, FP64, q, R, ws)
    ref = residual(osh.disc, osh.ph, Q)
    _, ev = rel_err(to5(R, p + 1), ref, W)
    assert np.all(ev <= 1e-12 * np.maximum(1.0, _condition(osh, Q, ref, W))), ev
    for scheme, name in ((0, "ssprk3"), (1, "ssprk54")):
        q, ws = state(FP32_PERT, torch.float32)
        m.rk_step_scheme(sh.params, FP32_PERT, scheme, q, ws, sh.dt, 1)
        ref = rk.run(osh.disc, osh.ph, Q, sh.dt, 1, scheme=name) - osh.background()
        e, ev = rel_err(to5(q, p + 1), ref, W)
        assert e < 1e-5, (name, ev)
    m.check()
