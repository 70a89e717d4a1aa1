"""The volume kernel's staging at the edges of its tiles, FP32 and FP64, every order.

Element counts that leave the last tile (4 to 14 elements) partly filled, or that are less than one
tile, against the oracle; and a state that starts off the 16-byte boundary of the bulk copies, which
the kernels then read with plain loads: the arithmetic is the same, so residual and RK steps have to
equal the aligned state's bit for bit.

Tolerance against the oracle: the library's own for the FP32 form, 1e-5 relative L2 per variable.
"""
import pytest

from chorus_inputs import small_shell
from gpu_common import OracleShell, rel_err, to5

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1503_00834_gb300 import build

    build.build()


# 6, 18, 24 and 30 elements; one-cell panels take a mild stratification (positive traces)
SHAPES = [(1, 1, 0.5), (1, 3, 0.5), (2, 1, 3.0), (1, 5, 0.5)]


@pytest.mark.parametrize("p", [2, 3, 4, 5])
@pytest.mark.parametrize("n, n_r, N_rho", SHAPES)
def test_partial_tiles_and_unaligned_state(p, n, n_r, N_rho):
    from oracle.residual import residual
    from paper_1503_00834_gb300 import FP32_PERT, FP64, Shell

    cfg = small_shell(n, n_r, p, N_rho=N_rho)
    sh = Shell(cfg)
    m = sh.mesh
    osh = OracleShell(cfg)
    for prec, dtype in ((FP32_PERT, torch.float32), (FP64, torch.float64)):
        q = torch.empty(m.state_shape(), dtype=dtype, device="cuda")
        m.state_init(sh.params, cfg.seed, cfg.entropy_amp, prec, q)
        ws = torch.empty(m.workspace_bytes(prec), dtype=torch.uint8, device="cuda")
        R = torch.empty_like(q)
        m.residual(sh.params, prec, q, R, ws)
        if prec == FP32_PERT:
            e, ev = rel_err(to5(R, p + 1), residual(osh.disc, osh.ph, osh.initial_state()), osh.weights())
            assert e < 1e-5, ev
        # the same state one word past a 16-byte boundary
        off = torch.empty(q.numel() + 1, dtype=dtype, device="cuda")[1:].view(q.shape)
        assert off.data_ptr() % 16 != 0
        off.copy_(q)
        R2 = torch.empty_like(q)
        m.residual(sh.params, prec, off, R2, ws)
        assert torch.equal(R2, R)
        for scheme in (0, 1):
            m.rk_step_scheme(sh.params, prec, scheme, q, ws, 0.1 * sh.dt, 2)
            m.rk_step_scheme(sh.params, prec, scheme, off, ws, 0.1 * sh.dt, 2)
            assert torch.equal(off, q)
        m.check()
