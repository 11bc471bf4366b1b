"""The FP64 form's Jacobian and gradient against sums in extended precision (long double), around and past the
width of 1024.  Linear layers, so that nothing but the products rounds.

Tolerance (relative Frobenius): operands of 54 bits or more cost no more than the rounding of a result to FP64,
whose size is at most 2^-53 / sqrt(3) in the mean over the entries.  Two such roundings for each of three
products, independent of each other: sqrt(6 / 3) 2^-53; and one constant of each product, rounded the same way
in every entry: 3 * 2^-53.  Together 4.9e-16."""
import numpy as np
import pytest

from synth.nets import MLPSpec, make_mlp
from synth.rng import derive_key, normal, uniform01

pytestmark = pytest.mark.gpu

LD = np.longdouble


@pytest.fixture(scope="module")
def lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_22462_gb300 import build, nnc
    build.build()
    return nnc


def product(W):
    """The matrix of a linear net in long double."""
    J = W[-1].astype(LD)
    for w in W[-2::-1]:
        J = J @ w.astype(LD)
    return J


@pytest.mark.parametrize("widths", [[30, 896, 896, 3], [30, 1000, 1000, 3], [30, 1025, 1025, 3],
                                    [24, 2048, 2048, 4], [700, 1100, 64, 2]])
def test_against_long_double(lib, widths):
    mlp = make_mlp(MLPSpec(widths, ["identity"] * 3), seed=widths[1], tag="acc")
    x, lam = uniform01(derive_key(1, "acc-x"), widths[0]), normal(derive_key(1, "acc-lam"), widths[-1])
    net = lib.Net.from_mlp(mlp, precision="fp64")
    assert net.fp64_residues
    _, g = net.hessian_lag(x, lam, want_grad=True)
    J = net.jacobian(x)
    net.free()
    Jo = product(mlp.W)
    go = lam.astype(LD) @ Jo
    for got, ref in ((J, Jo), (g, go)):
        err = float(np.sqrt(np.sum((got - ref) ** 2) / np.sum(ref ** 2)))
        print(f"[{widths}] {err:.2e}")
        assert err < 4.9e-16
