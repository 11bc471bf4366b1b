"""A net, a batch or a warm-start network that does not fit is refused with NNC_ERR_OOM, and the calls after
it, on objects that were there, are none the wiser."""
import numpy as np
import pytest

from synth.nets import MLPSpec, make_mlp
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


@pytest.mark.parametrize("kind", ["net", "batch", "warmstart"])
def test_refusal_leaves_no_error(lib, kind):
    import torch
    mlp = make_mlp(MLPSpec([20, 200, 3], ["tanh", "identity"]), seed=2, tag="oom")
    x = np.full(20, 0.3)
    net = lib.Net.from_mlp(mlp, precision="fp32")
    y, J = net.eval(x), net.jacobian(x)
    n = 3000
    w = [normal(derive_key(i, "oom-w"), n * n).reshape(n, n) / n for i in range(3)]
    b = [np.zeros(n)] * 3
    wide = [lib.Net([30, n, n, 1], ["tanh", "tanh", "identity"],
                    [w[0][:, :30], w[1], w[2][:1]], [b[0], b[1], b[2][:1]], "bf16") for _ in range(2)]
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (40 << 20), dtype=torch.uint8, device="cuda")
    try:
        with pytest.raises(lib.NNCError) as e:
            if kind == "net":
                lib.Net([n, n, n, 3], ["tanh", "tanh", "identity"], [w[0], w[1], w[2][:3]], None, "fp32")
            elif kind == "batch":
                lib.Batch(wide)
            else:
                lib.WarmStart([w[0], b[0], w[1], b[1], w[2], b[2]], precision="fp32")
        assert e.value.code == -5
        assert np.array_equal(net.eval(x), y) and np.array_equal(net.jacobian(x), J)
    finally:
        del hold
        torch.cuda.empty_cache()
