"""Sums over many split partials in the tensor-core forms: the Hessian of nets of few inputs (more than 16
parts of K, small blocks) and the reverse sweep of nets of more than 15 outputs (more than 16 parts of the
first layer's rows), at the edges of the 32-wide tiles, against the FP64 oracle.  Tolerances of the forms:
Jacobian 1e-3, Hessian 1e-2 (relative Frobenius); H is exactly symmetric."""
import numpy as np
import pytest

from synth.nets import MLPSpec, make_mlp
from synth.rng import derive_key, normal, uniform01
from oracle import nn as onn

pytestmark = pytest.mark.gpu

NETS = [
    ([5, 1100, 1030, 2], ["tanh", "tanh", "identity"]),
    ([31, 1500, 17], ["tanh", "tanh"]),
    ([33, 1100, 1100, 20], ["sigmoid", "tanh", "identity"]),
    ([64, 2100, 3], ["tanh", "softmax"]),
    ([117, 1280, 1280, 37], ["tanh", "tanh", "identity"]),
    ([129, 1153, 16], ["gelu", "identity"]),
]


@pytest.mark.parametrize("prec", ["bf16", "bf16x3"])
@pytest.mark.parametrize("case", range(len(NETS)))
def test_split_sums(case, prec):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_22462_gb300 import build, nnc
    build.build()
    widths, acts = NETS[case]
    mlp = make_mlp(MLPSpec(widths, acts), seed=case + 20, tag="splits", bias_std=0.2)
    x, lam = uniform01(derive_key(case, "sp-x"), widths[0]), normal(derive_key(case, "sp-lam"), widths[-1])
    net = nnc.Net.from_mlp(mlp, precision=prec)
    H, J = net.hessian_lag(x, lam), net.jacobian(x)
    H2 = net.hessian_lag(x, lam)
    net.free()
    _, Jo, Ho, _ = onn.all_outputs(mlp, x, lam)
    assert np.linalg.norm(J - Jo) < 1e-3 * np.linalg.norm(Jo)
    assert np.linalg.norm(H - Ho) < 1e-2 * np.linalg.norm(Ho)
    assert np.array_equal(H, H.T) and np.array_equal(H, H2)
