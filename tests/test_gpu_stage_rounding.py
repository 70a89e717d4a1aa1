"""An SSP-RK3 step rounds each stage's state once, from the whole residual.

Each stage is u_new = fl(c fl(dt R) + fl(a u^n + fl(b u))) with one rounding for every fl, where R is the
residual as chorus_residual returns it.  The test forms the three stages that way, exactly (rational
arithmetic, rounded at each fl), from the library's own residuals, and compares one step of the library.

Both sides use the same R: a difference is left only where the stage's traces, made beside the new state,
round otherwise than chorus_residual's own (a few in the last place of R, seldom in the state's).  At
least 95 % of the values have to be equal, and the others within two units in the last place of the
largest term; a state rounded a second time, before the end-point fluxes of its lines are added, differs
in a quarter or more of them.
"""
from fractions import Fraction

import numpy as np
import pytest

from chorus_inputs import small_shell

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1503_00834_gb300 import build

    build.build()


def _combine(a, b, c, dt, un, q, R):
    """The stage on numpy arrays of one type, each operation rounded to it once."""
    t = q.dtype.type
    a, b, c, dt = Fraction(float(t(a))), Fraction(float(t(b))), Fraction(float(t(c))), Fraction(float(t(dt)))

    def fl(x):
        return Fraction(float(t(float(x))))

    out = np.empty_like(q)
    for i, (u, x, r) in enumerate(zip(un.flat, q.flat, R.flat)):
        base = fl(b * Fraction(float(x)))
        if a:
            base = fl(a * Fraction(float(u)) + base)
        out.flat[i] = t(float(c * fl(dt * Fraction(float(r))) + base))
    return out


@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "fp32"])
@pytest.mark.parametrize("p", [2, 3, 4, 5])
def test_step_is_the_once_rounded_combination_of_residuals(p, prec):
    from paper_1503_00834_gb300 import Shell

    cfg = small_shell(2, 2, p)
    sh = Shell(cfg)
    m = sh.mesh
    dtype = torch.float64 if prec == 0 else torch.float32
    q = torch.empty(m.state_shape(), dtype=dtype, device="cuda")
    m.state_init(sh.params, cfg.seed, cfg.entropy_amp, prec, q)
    ws = torch.empty(m.workspace_bytes(prec), dtype=torch.uint8, device="cuda")
    m.rk_step(sh.params, prec, q, ws, sh.dt, 20)  # away from the start, where the momentum is zero
    un = q.cpu().numpy()
    s, largest = un, np.abs(un)
    R = torch.empty_like(q)
    for a, b in ((0.0, 1.0), (0.75, 0.25), (1.0 / 3.0, 2.0 / 3.0)):
        m.residual(sh.params, prec, torch.tensor(s, device="cuda"), R, ws)
        Rh = R.cpu().numpy()
        largest = np.maximum(largest, np.maximum(np.abs(s), np.abs(Rh) * sh.dt))
        s = _combine(a, b, b, sh.dt, un, s, Rh)
    m.rk_step(sh.params, prec, q, ws, sh.dt, 1)
    m.check()
    got = q.cpu().numpy()
    ulp = np.spacing(largest)
    assert np.all(np.abs(got - s) <= 2 * ulp), float((np.abs(got - s) / ulp).max())
    equal = np.mean(got == s)
    print(f"p = {p}: {equal:.4f} of the values equal")
    assert equal >= 0.95
