"""Which products an FP64 net has: by residues on the tensor cores, or FP64 ones where the residues would
take more than an eighth of the free memory or the weights are uneven.  Results against the oracle at the
tolerance of the residue products (relative Frobenius 1e-12)."""
import numpy as np
import pytest

from synth.nets import MLPSpec, make_mlp
from synth.rng import derive_key, normal, uniform01
from oracle import nn as onn

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_22462_gb300 import build, nnc
    build.build()
    return nnc


def load(lib, mlp, precision="fp64"):
    """(by residues?, device memory that the net takes) after checking its outputs."""
    import torch
    n, m = mlp.spec.widths[0], mlp.spec.widths[-1]
    x, lam = uniform01(derive_key(1, "route-x"), n), normal(derive_key(1, "route-lam"), m)
    free = torch.cuda.mem_get_info()[0]
    net = lib.Net.from_mlp(mlp, precision=precision)
    taken = free - torch.cuda.mem_get_info()[0]
    by_residues = net.fp64_residues
    if precision == "fp64":
        H, g = net.hessian_lag(x, lam, want_grad=True)
        J = net.jacobian(x)
        _, Jo, Ho, go = onn.all_outputs(mlp, x, lam)
        for a, b in ((J, Jo), (H, Ho), (g, go)):
            assert np.linalg.norm(a - b) < 1e-12 * np.linalg.norm(b)
    net.free()
    return by_residues, taken


@pytest.fixture(scope="module")
def mlp():
    return make_mlp(MLPSpec([300, 140, 130, 3], ["tanh", "gelu", "softmax"]), seed=6, tag="route")


def test_forms(lib, mlp):
    assert load(lib, mlp)[0]
    assert not load(lib, mlp, "fp32")[0] and not load(lib, mlp, "bf16")[0]


def test_uneven_weights_free_their_residues(lib, mlp):
    pruned = make_mlp(mlp.spec, seed=7, tag="route")
    pruned.W[1][:, ::3] *= 2.0 ** -12     # evened out by powers of two
    assert load(lib, pruned)[0]
    keep = uniform01(derive_key(2, "route-keep"), pruned.W[1].size).reshape(pruned.W[1].shape) < 0.5
    pruned.W[1] *= keep                   # half of the weights are zero
    by_residues, taken = load(lib, pruned)
    assert not by_residues and taken < load(lib, mlp)[1]


def test_share_of_the_free_memory(lib, mlp):
    import torch
    torch.cuda.empty_cache()
    by_residues, size = load(lib, mlp)
    assert by_residues and size > 16 << 20
    for room, expected in ((4, False), (16, True)):
        hold = torch.empty(torch.cuda.mem_get_info()[0] - room * size, dtype=torch.uint8, device="cuda")
        try:
            by_residues, taken = load(lib, mlp)
            assert by_residues == expected
            assert taken < size / 2 or expected
        finally:
            del hold
            torch.cuda.empty_cache()
