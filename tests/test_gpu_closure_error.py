"""Error of the closure gradient against 64 bits, over the sizes at which the tile changes.

A tile's share of the gradient is summed in FP32 and added to the result with atomics, each addition
rounded once.  With m tiles of 32 samples the running sum reaches j/m of its end after j of them, so the
additions leave a relative error of u sqrt(m / 3), u = 2.4e-8 the rms rounding error of one FP32 addition
(2^-23 / sqrt(12) of the last place, times the rms of 1/x over a binade, 0.71).  What the network and the
sums inside the tiles contribute is measured: the same gradient put together in 64 bits from calls of one
tile each.  Bound: both together, with 1.2 times the model for the additions.  Twice as many additions
(tiles of 16 samples) are 1.41 times the model.
"""
import numpy as np
import pytest

from test_gpu_closure import IN_SCALE, OUT_SCALE, _oracle_params

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TILE = 32


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1503_00834_gb300 import build

    build.build()


@pytest.mark.parametrize("n", [1024, 2400, 4832, 4896])
def test_gradient_error_is_that_of_its_tiles(n):
    from oracle.closure import loss_and_grad
    from paper_1503_00834_gb300 import native

    w = native.closure_alloc(7, IN_SCALE, OUT_SCALE)
    rng = np.random.default_rng(n)
    X = rng.uniform(-1.0, 1.0, (n, 135)).astype(np.float32)
    T = (0.5 * np.tanh(np.roll(X, 3, 1)) + 0.1 * rng.uniform(0.0, 1.0, X.shape)).astype(np.float32)
    _, g = loss_and_grad(_oracle_params(w), X.astype(np.float64), T.astype(np.float64))
    exact = np.concatenate([g[k].reshape(-1) for k in ("W1", "W2", "W3", "b1", "b2", "b3")])
    Xd, Td = torch.tensor(X, device="cuda"), torch.tensor(T, device="cuda")
    out = torch.empty(native.N_PARAMS, dtype=torch.float32, device="cuda")

    def err(grad):
        return np.linalg.norm(grad - exact) / np.linalg.norm(exact)

    tiles = np.zeros(native.N_PARAMS)
    for r in range(0, n, TILE):
        native.closure_grad(w, Xd[r:r + TILE].contiguous(), Td[r:r + TILE].contiguous(), out)
        tiles += out.cpu().numpy().astype(np.float64) * (TILE / n)
    got = []
    for _ in range(8):  # the order of the additions differs from call to call
        native.closure_grad(w, Xd, Td, out)
        got.append(err(out.cpu().numpy().astype(np.float64)))
    bound = np.hypot(err(tiles), 1.2 * 2.4e-8 * np.sqrt(n / TILE / 3.0))
    print(f"{n}: error {np.mean(got):.3e}, tiles {err(tiles):.3e}, bound {bound:.3e}")
    assert np.mean(got) <= bound
