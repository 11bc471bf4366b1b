"""Host calls of small nets bring their pageable outputs through one pinned block (up to 256 KB: 179 inputs
and 3 outputs): bit for bit what the device call writes, on both sides of that size, for every form, and when
some of the outputs are page-locked themselves."""
import numpy as np
import pytest

from synth.nets import MLPSpec, make_mlp
from synth.rng import derive_key, normal, uniform01

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("n", [1, 178, 179, 180])
def test_staged_outputs(n, prec):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_22462_gb300 import build, nnc
    build.build()
    mlp = make_mlp(MLPSpec([n, 70, 65, 3], ["tanh", "gelu", "identity"]), seed=n, tag="staged", bias_std=0.2)
    net = nnc.Net.from_mlp(mlp, precision=prec)
    x = uniform01(derive_key(n, "st-x"), n)
    y, lam = normal(derive_key(n, "st-y"), 3), normal(derive_key(n, "st-lam"), 3)
    dev = [torch.empty(*s, device="cuda", dtype=torch.float64) for s in ((3,), (3, n), (n, n), (n,))]
    r, J, H, g = dev
    args = [torch.from_numpy(v).cuda() for v in (x, y, lam)]
    net.eval_kkt_dev(args[0], y=args[1], lam=args[2], r=r, J=J, H=H, grad=g)
    torch.cuda.synchronize()
    want = [t.cpu().numpy() for t in dev]
    for _ in range(2):
        got = net.eval_kkt(x, y, lam)
        assert all(np.array_equal(a, b) for a, b in zip(got, want))
    pinned = [torch.empty(*t.shape, dtype=torch.float64, pin_memory=True).numpy() for t in dev]
    mixed = [pinned[0], np.empty((3, n)), pinned[2], np.empty(n)]
    got = net.eval_kkt(x, y, lam, out=mixed)
    assert all(np.array_equal(a, b) for a, b in zip(got, want))
    yv, Jv = net.eval(x), net.jacobian(x)
    assert np.array_equal(Jv, want[1]) and np.allclose(yv, y - want[0], rtol=0, atol=1e-12)
    net.free()
