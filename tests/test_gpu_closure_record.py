"""Closure records that start on a 4-byte boundary only.

The record's fields are BF16 and FP32, so any 4-byte-aligned address holds one (a slice of a larger
buffer, for instance).  The kernels' wider loads have to look at the address: results from a record at
4, 8 and 12 bytes past a 16-byte boundary against those from an aligned copy, for the three tile sizes
of the FP32 kernels (by the number of samples) and for the tensor-core kernel.

Tolerances: the forward passes do the same arithmetic, so they have to agree bit for bit; gradients and
loss are sums of the same products in the order in which the CTAs arrive, each CTA's share rounded in
FP32: 1e-5 relative.
"""
import numpy as np
import pytest

from test_gpu_closure import IN_SCALE, OUT_SCALE

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1503_00834_gb300 import build

    build.build()


def _shifted(w, off):
    buf = torch.zeros(w.numel() + 16, dtype=torch.uint8, device="cuda")
    s = buf[off:off + w.numel()]
    s.copy_(w)
    assert s.data_ptr() % 16 == off
    return s


@pytest.mark.parametrize("off", [4, 8, 12])
@pytest.mark.parametrize("n", [17, 2433, 4865])
def test_forward_gradient_and_training(n, off):
    from paper_1503_00834_gb300 import native

    w = native.closure_alloc(11, IN_SCALE, OUT_SCALE)
    s = _shifted(w, off)
    rng = np.random.default_rng(n)
    X = torch.tensor(rng.standard_normal((n, 135)).astype(np.float32), device="cuda")
    T = torch.tensor((0.3 * rng.standard_normal((n, 135))).astype(np.float32), device="cuda")
    for forward in (native.closure_forward, native.closure_forward_tc):
        Y, Z = torch.empty_like(X), torch.empty_like(X)
        forward(w, X, Y)
        forward(s, X, Z)
        assert torch.equal(Y, Z)
    g = [torch.empty(native.N_PARAMS, dtype=torch.float32, device="cuda") for _ in range(2)]
    loss = [native.closure_grad(r, X, T, gr) for r, gr in zip((w, s), g)]
    assert abs(loss[1] - loss[0]) <= 1e-5 * loss[0]
    assert (g[1] - g[0]).norm() <= 1e-5 * g[0].norm()
    # the first epoch is the untrained record's loss; one Adam step of 1e-3 then lowers it (lr |g|_1 to
    # first order)
    losses = native.closure_train(X, T, s, epochs=2, batch=n, lr=1e-3)
    assert abs(losses[0] - loss[0]) <= 1e-5 * loss[0]
    assert losses[1] < losses[0]
