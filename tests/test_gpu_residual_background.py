"""At p = 2 the FP32 residual adds R(Q0) to a finished perturbation residual, with one rounding.

A coarse p = 2 shell's residual is mostly R(Q0), so a rounding more at its size shows.
chorus_set_well_balanced leaves R(Q0) out, so the full residual has to be fl(R_wb + R(Q0)) of the two.
R(Q0) is the FP64 residual of the unperturbed state rounded to FP32; the library's own table comes from
other FP64 kernels, whose rounding (1e-13 relative) can move a value across an FP32 rounding boundary in
about one of 1e5.  At least 99.9 % of the values have to be equal; where R(Q0) enters before the end-point
fluxes of the lines, one in five or more differs.
"""
import pytest

from chorus_inputs import small_shell

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n, n_r", [(3, 2), (4, 3), (5, 3)])
def test_full_residual_is_the_rounded_sum(n, n_r):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1503_00834_gb300 import FP32_PERT, FP64, Shell, build

    build.build()
    cfg = small_shell(n, n_r, 2)
    sh = Shell(cfg)
    m = sh.mesh
    Q = torch.empty(m.state_shape(), dtype=torch.float64, device="cuda")
    m.state_init(sh.params, cfg.seed, 0.0, FP64, Q)
    R0 = torch.empty_like(Q)
    m.residual(sh.params, FP64, Q, R0, torch.empty(m.workspace_bytes(FP64), dtype=torch.uint8, device="cuda"))
    q = torch.empty(m.state_shape(), dtype=torch.float32, device="cuda")
    m.state_init(sh.params, cfg.seed, cfg.entropy_amp, FP32_PERT, q)
    ws = torch.empty(m.workspace_bytes(FP32_PERT), dtype=torch.uint8, device="cuda")
    m.rk_step(sh.params, FP32_PERT, q, ws, sh.dt, 5)
    full, wb = torch.empty_like(q), torch.empty_like(q)
    m.residual(sh.params, FP32_PERT, q, full, ws)
    m.set_well_balanced(True)
    m.residual(sh.params, FP32_PERT, q, wb, ws)
    m.set_well_balanced(False)
    m.check()
    equal = (full == wb + R0.float()).double().mean().item()
    print(f"{n} x {n_r}: {equal:.5f} equal")
    assert equal >= 0.999
