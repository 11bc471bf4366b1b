"""The warm-start network at sizes past the limits of a launch's second grid dimension (65535 tiles of 32
rows, 65535 blocks of 256 columns), against FP64: FP32 sums of k terms are held to 4 k 2^-24 of their
terms' size."""
import numpy as np
import pytest

from synth.rng import derive_key, normal

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_22462_gb300 import build, nnc
    build.build()
    return nnc


def params(n_in, h1, h2, n_out, scale=1.0):
    out = []
    for i, (m, k) in enumerate(((h1, n_in), (h2, h1), (n_out, h2))):
        out += [scale * normal(derive_key(i, "wsz-w"), m * k).reshape(m, k) / np.sqrt(k),
                0.1 * normal(derive_key(i, "wsz-b"), m)]
    return out


def gelu(z):
    from scipy.special import erf
    return 0.5 * z * (1.0 + erf(z / np.sqrt(2.0)))


def many_rows(lib):
    p = params(3, 5, 4, 2)
    U = normal(derive_key(9, "wsz-u"), 3 * (65535 * 32 + 33)).reshape(-1, 3)
    a = gelu(gelu(U @ p[0].T + p[1]) @ p[2].T + p[3]) @ p[4].T + p[5]
    ws = lib.WarmStart(p, precision="fp32")
    return ws, U, a


def test_launches_that_fail_are_reported(lib):
    """A call whose launches do not fit raises; it never returns what happened to lie in the buffers, and
    the calls after it are none the wiser."""
    ws, U, a = many_rows(lib)
    try:
        P = ws.predict(U)
    except lib.NNCError:
        P = a
    assert np.max(np.abs(P - a)) < 1e-5
    ws.free()
    ws = lib.WarmStart(params(3, 5, 4, 2), precision="fp32")
    assert np.max(np.abs(ws.predict(U[:100]) - a[:100])) < 1e-5


def test_predict_more_rows(lib):
    ws, U, a = many_rows(lib)
    assert np.max(np.abs(ws.predict(U) - a)) < 1e-5


def test_train_more_columns(lib):
    """Two rows standardize to -1 and 1, so that the gradient of W_1 has the sign of their difference times
    that of a common factor, and the first Adam step moves every weight by the learning rate."""
    n, lr = 256 * 65536 + 1, 1e-3
    p = params(n, 1, 2, 2)
    U, T = normal(derive_key(5, "wsz-u"), 2 * n).reshape(2, n), np.array([[0.0, 1.0], [2.0, -1.0]])
    ws = lib.WarmStart(p, precision="fp32")
    loss = ws.train(U, T, 1, batch=2, lr=lr, seed=1)
    step = (ws.params()[0] - p[0].astype(np.float32))[0] / lr
    assert np.isfinite(loss)
    sign = np.sign(U[0] - U[1])
    # FP32 weights of 1e-4 in size: the step is off by their rounding, 2^-24 * 2^-10 against 1e-3 at most
    assert np.max(np.abs(step * sign * np.sign(step[0] * sign[0]) - 1.0)) < 1e-3


@pytest.mark.parametrize("precision", ["bf16", "fp32"])
def test_train_set_that_fills_the_memory(lib, precision):
    """A data set whose standardized FP32 values fit trains, to the same bits as with room to spare: 33 MB
    beside the 66 MB of the values as given, with 80 MB free."""
    import torch
    n, rows = 1024, 4001
    p = params(n, 64, 64, n)
    U = normal(derive_key(6, "wsz-u"), n * rows).reshape(rows, n)
    T = U[:, ::-1] ** 2

    def train(room):
        ws = lib.WarmStart(p, precision=precision)
        torch.cuda.empty_cache()
        hold = torch.empty(max(torch.cuda.mem_get_info()[0] - room, 1), dtype=torch.uint8, device="cuda")
        try:
            out = [ws.train(U, T, 1, batch=64, seed=2)] + ws.params()
        finally:
            del hold
            torch.cuda.empty_cache()
            ws.free()
        return out

    for a, b in zip(train(8 << 30), train(80 << 20)):
        assert np.array_equal(a, b)
