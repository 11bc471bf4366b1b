"""The FP64 form on nets of uneven scale, column by column: inputs and hidden units many powers of two
apart, and weights that no scaling of rows and columns evens out.

Tolerance, relative to each column: rows and columns of the even nets below have their largest entry
within 8 rms, the powers of two that even them out are right to a factor of two, and four products of
operands rounded to 52 bits of their largest entry follow one another: 4 * 32 * 2^-52 = 2.8e-14 in size,
against which sums that cancel lose up to a factor of 30: 1e-12.
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


def evaluate(lib, mlp, x, lam):
    net = lib.Net.from_mlp(mlp, precision="fp64")
    H, g = net.hessian_lag(x, lam, want_grad=True)
    J = net.jacobian(x)
    net.free()
    return J, H, g


def columns(a, b):
    """Largest relative error of a column of a against b."""
    return float(np.max(np.linalg.norm(a - b, axis=0) / np.linalg.norm(b, axis=0)))


def check(lib, mlp, x, lam, s=None):
    """J, H and g of mlp against the oracle; s: the inputs' scales, divided out."""
    s = np.ones(x.size) if s is None else s
    J, H, g = evaluate(lib, mlp, x, lam)
    _, Jo, Ho, go = onn.all_outputs(mlp, x, lam)
    size = (np.abs(lam) @ np.abs(Jo)) / s   # what the gradient's terms add up to
    assert columns(J / s, Jo / s) < TOL
    assert np.max(np.abs(g - go) / s / size) < TOL
    assert columns(H / np.outer(s, s), Ho / np.outer(s, s)) < TOL
    return J


def powers(key, n, spread):
    """n powers of two, spread over 2^spread around 1."""
    return 2.0 ** np.round(spread * (uniform01(derive_key(key, "scale-t"), n) - 0.5))


def point(n, m, key):
    return uniform01(derive_key(key, "scale-x"), n), normal(derive_key(key, "scale-lam"), m)


NETS = [([60, 200, 150, 4], ["tanh", "sigmoid", "identity"]),
        ([33, 129, 65, 5], ["gelu", "tanh", "softmax"]),
        ([300, 1500, 1100, 3], ["tanh", "tanh", "identity"]),
        ([90, 4], ["tanh"])]


@pytest.mark.parametrize("spread", [20, 40, 60])
@pytest.mark.parametrize("case", range(len(NETS)))
def test_input_scales(lib, case, spread):
    """Inputs in units of their own: W_1 times s by column at x / s is the same function."""
    widths, acts = NETS[case]
    mlp = make_mlp(MLPSpec(widths, acts), seed=case + 20, tag="scales", bias_std=0.1)
    x, lam = point(widths[0], widths[-1], case)
    s = powers(case, widths[0], spread)
    scaled = MLP(mlp.spec, [mlp.W[0] * s[None, :]] + list(mlp.W[1:]), mlp.b)
    check(lib, scaled, x / s, lam, s)


@pytest.mark.parametrize("spread", [20, 40])
@pytest.mark.parametrize("width", [150, 1100])
def test_linear_unit_scales(lib, width, spread):
    """Units of a linear hidden layer times t, taken back by the next layer's columns."""
    widths, acts = [50, 180, width, 140, 3], ["tanh", "identity", "sigmoid", "identity"]
    mlp = make_mlp(MLPSpec(widths, acts), seed=31, tag="scales", bias_std=0.1)
    t = powers(width, width, spread)
    W, b = list(mlp.W), list(mlp.b)
    W[1], b[1], W[2] = W[1] * t[:, None], b[1] * t, W[2] / t[None, :]
    check(lib, MLP(mlp.spec, W, b), *point(50, 3, 31))


@pytest.mark.parametrize("spread", [20, 40])
@pytest.mark.parametrize("case", range(3))
def test_hidden_unit_scales(lib, case, spread):
    """Units of curved hidden layers scaled down by 1 .. 2^-spread, the next layer's columns up."""
    widths, acts = NETS[case]
    mlp = make_mlp(MLPSpec(widths, acts), seed=case + 40, tag="scales", bias_std=0.1)
    t = powers(case + 7, widths[1], spread) * 2.0 ** -(spread // 2)
    W, b = list(mlp.W), list(mlp.b)
    W[0], b[0], W[1] = W[0] * t[:, None], b[0] * t, W[1] / t[None, :]
    check(lib, MLP(mlp.spec, W, b), *point(widths[0], widths[-1], case + 40))


def test_output_scales(lib):
    """Outputs many powers of two apart: every row of J keeps its own accuracy."""
    mlp = make_mlp(MLPSpec([40, 130, 120, 12], ["tanh", "sigmoid", "identity"]), seed=5, tag="scales")
    t = powers(5, 12, 40)
    mlp.W[2] *= t[:, None]
    x, lam = point(40, 12, 5)
    J = check(lib, mlp, x, lam)
    assert columns(J.T / t, onn.all_outputs(mlp, x, lam)[1].T / t) < TOL


def uneven(kind, m, k, key):
    """Weights whose rows and columns no powers of two even out."""
    W = normal(derive_key(key, "scale-w"), m * k).reshape(m, k) / np.sqrt(k)
    t = 2.0 ** -30
    if kind == "blocks":       # two groups of units, weakly coupled
        W[: m // 2, k // 2:] *= t
        W[m // 2:, : k // 2] *= t
    elif kind == "entries":    # every entry a power of two of its own
        W *= powers(key + 1, m * k, 40).reshape(m, k) * 2.0 ** -20
    elif kind == "outlier":    # one entry far above its row and column
        W[m // 3, k // 3] /= t
    elif kind == "diagonal":   # groups that do not meet at all
        W[: m // 2, k // 2:] = 0.0
        W[m // 2:, : k // 2] = 0.0
    elif kind == "tiny":       # outside of the range in which scales are exact
        W[:, k // 2:] *= 2.0 ** -300
    return W


@pytest.mark.parametrize("kind", ["blocks", "entries", "outlier", "diagonal", "tiny"])
@pytest.mark.parametrize("layer", [0, 1])
def test_uneven_weights(lib, kind, layer):
    """FP64 products keep the accuracy of each column where residues of a row cannot.  Sums of terms of
    one sign (the activations' slopes are positive, and so are the weights here), so that no column
    cancels and the tolerance holds without its factor of 30."""
    widths, acts = [48, 160, 144, 3], ["softplus", "softplus", "identity"]
    mlp = make_mlp(MLPSpec(widths, acts), seed=9, tag="scales", bias_std=0.1)
    W = [np.abs(w) for w in mlp.W]
    W[layer] = np.abs(uneven(kind, widths[layer + 1], widths[layer], 50 + layer))
    if kind in ("blocks", "diagonal"):
        W[layer + 1][:, widths[layer + 1] // 2:] *= 2.0 ** -30   # the second group matters less
    x, lam = uniform01(derive_key(3, "scale-x"), 48), 0.5 + uniform01(derive_key(3, "scale-lam"), 3)
    if kind == "outlier":
        x = x * 2.0 ** -30     # keeps the activations in range
    check(lib, MLP(mlp.spec, W, mlp.b), x, lam)


@pytest.mark.parametrize("n", [2, 3, 6, 15])
def test_outlier_of_few_inputs(lib, n):
    """One weight far above the others of a short row: too few entries to count, and the row's scale would
    push the seeds of all other rows down."""
    mlp = make_mlp(MLPSpec([n, 160, 144, 3], ["softplus", "softplus", "identity"]), seed=n, tag="scales", bias_std=0.1)
    W = [np.abs(w) for w in mlp.W]
    W[0][53, n // 3] *= 2.0 ** 30
    x, lam = uniform01(derive_key(n, "scale-x"), n) * 2.0 ** -30, 0.5 + uniform01(derive_key(n, "scale-lam"), 3)
    check(lib, MLP(mlp.spec, W, mlp.b), x, lam)
