"""The closure kernels at the edges of their tiles and of the dispatch between tile sizes.

Gradient and FP32 forward: 16, 32 or 64 samples per CTA by the number of samples (16 below 2,432, 64
from 4,864); tensor-core forward: tiles of 128, several per CTA from 152 tiles on.  Against the FP64
oracle (network and backpropagation), tolerances as for the same quantities in test_gpu_closure.py:
forward 1e-5 (FP32) and 1e-4 (tensor cores, oracle with the same BF16 roundings), gradient 1e-4, loss
1e-5 relative.
"""
import threading

import numpy as np
import pytest

from test_gpu_closure import IN_SCALE, OUT_SCALE, _oracle_params

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1503_00834_gb300 import build

    build.build()


def _samples(n, seed):
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((n, 135)).astype(np.float32)
    T = (0.3 * rng.standard_normal((n, 135))).astype(np.float32)
    return X, T, torch.tensor(X, device="cuda"), torch.tensor(T, device="cuda")


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("n", [1, 15, 16, 17, 2431, 2432, 2433, 4863, 4864, 4865])
def test_gradient_and_forward(n):
    from oracle.closure import forward, loss_and_grad
    from paper_1503_00834_gb300 import native

    w = native.closure_alloc(7, IN_SCALE, OUT_SCALE)
    p = _oracle_params(w)
    X, T, Xd, Td = _samples(n, n)
    Yd = torch.empty_like(Xd)
    native.closure_forward(w, Xd, Yd)
    assert _rel(Yd.cpu().numpy(), forward(p, X.astype(np.float64))[0]) < 1e-5
    lref, gref = loss_and_grad(p, X.astype(np.float64), T.astype(np.float64))
    flat = np.concatenate([gref[k].reshape(-1) for k in ("W1", "W2", "W3", "b1", "b2", "b3")])
    buf = torch.empty(native.N_PARAMS + 1, dtype=torch.float32, device="cuda")
    for g in (buf[:-1], buf[1:]):  # 16-byte aligned (vector atomics) and not
        loss = native.closure_grad(w, Xd, Td, g)
        assert abs(loss - lref) < 1e-5 * lref
        assert _rel(g.cpu().numpy(), flat) < 1e-4


@pytest.mark.parametrize("n", [127, 128, 129, 152 * 128, 152 * 128 + 1, 2 * 152 * 128 + 77])
def test_tensor_core_tiles(n):
    from oracle.closure import forward_bf16_inputs
    from paper_1503_00834_gb300 import native

    w = native.closure_alloc(9, IN_SCALE, OUT_SCALE)
    X, _, Xd, _ = _samples(n, n)
    Yd = torch.full_like(Xd, float("nan"))
    native.closure_forward_tc(w, Xd, Yd)
    assert _rel(Yd.cpu().numpy(), forward_bf16_inputs(_oracle_params(w), X.astype(np.float64))) < 1e-4


def test_gradient_calls_from_several_threads_and_streams():
    """Each call has a loss word of its own while it runs."""
    from paper_1503_00834_gb300 import native

    w = native.closure_alloc(7, IN_SCALE, OUT_SCALE)
    data = [_samples(64 * (i + 1), i)[2:] for i in range(4)]
    grads = [torch.empty(native.N_PARAMS, dtype=torch.float32, device="cuda") for _ in data]
    want = [native.closure_grad(w, X, T, g) for (X, T), g in zip(data, grads)]
    torch.cuda.synchronize()
    bad = []

    def loop(i):
        stream = torch.cuda.Stream()
        for _ in range(50):
            got = native.closure_grad(w, *data[i], grads[i], stream=stream.cuda_stream)
            if abs(got - want[i]) > 1e-12 * want[i]:
                bad.append((i, got, want[i]))

    threads = [threading.Thread(target=loop, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
