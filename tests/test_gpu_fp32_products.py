"""The FP32 form's products (csrc/k_simt.cu: k_sgemm) against the FP64 oracle at the edges of their tiles
and where the tile changes: one tangent, tangent counts next to multiples of 32 and 64, widths next to
multiples of 128, one and several parts of K in the symmetric product.

Tolerance (relative Frobenius): a sum of K FP32 products in order is off by at most K 2^-24 of its terms'
size, here K <= 1152: 7e-5; two follow one another, and sums that cancel lose up to a factor of 10 here:
1.4e-3.  A misplaced or missing element gives an error of order one over the row's length, above 1e-2.
"""
import numpy as np
import pytest

from synth.nets import MLPSpec, make_mlp
from synth.rng import derive_key, normal, uniform01
from oracle import nn as onn

pytestmark = pytest.mark.gpu

NETS = [
    ([1, 128, 128, 1], ["tanh", "tanh", "identity"]),
    ([31, 64, 65, 2], ["sigmoid", "tanh", "identity"]),
    ([33, 129, 127, 3], ["gelu", "tanh", "softmax"]),
    ([64, 1, 200, 4], ["tanh", "softplus", "identity"]),
    ([65, 1100, 1030, 5], ["tanh", "tanh", "identity"]),
    ([257, 384, 300, 20], ["tanh", "identity", "tanh"]),
    ([784, 512, 1024, 10], ["sigmoid", "tanh", "softmax"]),
]


@pytest.mark.parametrize("case", range(len(NETS)))
def test_shapes(case):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_22462_gb300 import build, nnc
    build.build()
    widths, acts = NETS[case]
    mlp = make_mlp(MLPSpec(widths, acts), seed=case + 40, tag="sgemm", bias_std=0.2)
    x, lam = uniform01(derive_key(case, "sg-x"), widths[0]), normal(derive_key(case, "sg-lam"), widths[-1])
    net = nnc.Net.from_mlp(mlp, precision="fp32")
    H, H2 = net.hessian_lag(x, lam), net.hessian_lag(x, lam)
    net.free()
    Ho = onn.all_outputs(mlp, x, lam)[2]
    assert np.linalg.norm(H - Ho) < 1.4e-3 * np.linalg.norm(Ho)
    assert np.array_equal(H, H.T) and np.array_equal(H, H2)
