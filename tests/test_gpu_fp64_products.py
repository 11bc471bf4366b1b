"""The FP64 form's residue products (csrc/k_rns.cu) against the FP64 oracle at the sizes where they
change shape: the edges of tiles and column blocks, 16 and 15 moduli, one and several exact
accumulations of 1024 terms, 16, 32 and 48 seed columns, softmax columns, and the CUDA-core products
that stay where the residues do not fit in memory.

Tolerance (relative Frobenius).  Every row of an operand is rounded to 52 bits or more of its largest
entry, so a product is off by at most 2 * 2^-52 * t of its terms' size, t = largest / rms entry of a
row (t < 8 for these nets), and at most four products follow one another: 4 * 16 * 2^-52 = 1.4e-14
in size, against which sums that cancel lose up to a factor of 30 here: 1e-12.  One wrong residue gives
an error of order one.
"""
import numpy as np
import pytest

from synth.nets import MLP, MLPSpec, make_mlp
from synth.rng import derive_key, normal, uniform01
from oracle import nn as onn

pytestmark = pytest.mark.gpu

TOL = 1e-12


@pytest.fixture(scope="module")
def lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_22462_gb300 import build, nnc
    build.build()
    return nnc


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - b) / max(np.linalg.norm(b), 1e-300))


def check(lib, mlp, seed):
    n, m = mlp.spec.widths[0], mlp.spec.widths[-1]
    x, lam = uniform01(derive_key(seed, "rns-x"), n), normal(derive_key(seed, "rns-lam"), m)
    net = lib.Net.from_mlp(mlp, precision="fp64")
    H, g = net.hessian_lag(x, lam, want_grad=True)
    H2 = net.hessian_lag(x, lam)
    J = net.jacobian(x)
    net.free()
    yo, Jo, Ho, go = onn.all_outputs(mlp, x, lam)
    assert rel(J, Jo) < TOL and rel(g, go) < TOL
    assert rel(H, Ho) < TOL, rel(H, Ho)
    assert np.array_equal(H, H.T) and np.array_equal(H, H2)


NETS = [
    ([1, 128, 128, 1], ["tanh", "tanh", "identity"]),
    ([16, 129, 1, 3], ["sigmoid", "gelu", "tanh"]),
    ([208, 256, 255, 4], ["tanh", "softplus", "identity"]),
    ([209, 127, 384, 15], ["gelu", "identity", "softmax"]),
    ([257, 1023, 1025, 2], ["tanh", "tanh", "identity"]),
    ([40, 2049, 1152, 47], ["sigmoid", "tanh", "softmax"]),
    ([1025, 200, 16], ["tanh", "identity"]),
    ([130, 33], ["softmax"]),
    ([12, 7], ["tanh"]),
    ([5] + [8] * 66 + [2], ["tanh"] * 66 + ["identity"]),
]


@pytest.mark.parametrize("case", range(len(NETS)))
def test_shapes(lib, case):
    widths, acts = NETS[case]
    check(lib, make_mlp(MLPSpec(widths, acts), seed=case + 90, tag="rns", bias_std=0.2), case)


@pytest.mark.parametrize("k", [1024, 3072])
def test_equal_entries(lib, k):
    """Rows of equal entries: the residues of a row agree, so the sums reach the largest values that
    the exact accumulation has to hold."""
    widths, acts = [24, k, k, 3], ["tanh", "tanh", "identity"]
    W = [np.outer(0.3 + uniform01(derive_key(l, "rns-eq"), widths[l + 1]), np.ones(widths[l])) / widths[l]
         for l in range(3)]
    check(lib, MLP(MLPSpec(widths, acts), W, [np.zeros(w) for w in widths[1:]]), 7)


def test_row_scales(lib):
    """Rows and inputs whose sizes lie many powers of two apart keep their own accuracy: H of a net
    with scaled inputs is the scaled H."""
    mlp = make_mlp(MLPSpec([60, 200, 150, 4], ["tanh", "sigmoid", "identity"]), seed=3, tag="rns-scale")
    s = 2.0 ** np.round(40 * (uniform01(derive_key(1, "rns-s"), 60) - 0.5))
    x, lam = uniform01(derive_key(2, "rns-x"), 60), normal(derive_key(2, "rns-lam"), 4)
    net = lib.Net.from_mlp(mlp, precision="fp64")
    H = net.hessian_lag(x, lam)
    net.free()
    W = [mlp.W[0] * s[None, :]] + mlp.W[1:]
    net = lib.Net(mlp.spec.widths, mlp.spec.acts, W, mlp.b, "fp64")
    Hs = net.hessian_lag(x / s, lam)
    net.free()
    assert np.array_equal(Hs / np.outer(s, s), H)   # powers of two: not one bit differs


def test_no_room_for_residues(lib):
    """With little free memory the net keeps the CUDA-core products."""
    import torch
    mlp = make_mlp(MLPSpec([300, 140, 130, 3], ["tanh", "gelu", "softmax"]), seed=5, tag="rns-room")
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    hold = torch.empty(free - (48 << 20), dtype=torch.uint8, device="cuda")   # residues need 31 of 24
    try:
        check(lib, mlp, 5)
    finally:
        del hold
        torch.cuda.empty_cache()
    check(lib, mlp, 5)


def test_nan_weight(lib):
    """A NaN in the weights shows in H, as in any FP64 arithmetic."""
    mlp = make_mlp(MLPSpec([20, 64, 64, 2], ["tanh", "tanh", "identity"]), seed=4, tag="rns-nan")
    mlp.W[1][5, 7] = np.nan
    net = lib.Net.from_mlp(mlp, precision="fp64")
    H = net.hessian_lag(np.full(20, 0.5), np.ones(2))
    net.free()
    assert np.isnan(H).all()
