"""The streaming value pass at its edges: one to sixteen warps per row, with and without the warp that
finishes the rows, one row to four batches of 32 rows per CTA.  Residual y - NN(x) against FP64 products
on the host: 1e-10 max(1, |y|), the tolerance of every form; evaluations take the same values."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHAPES = [
    [1, 1, 1],               # one row, one column
    [511, 33, 2],            # one warp
    [1025, 513, 97, 3],      # three warps, then two, then one
    [1537, 456, 4],          # four warps and the finishing one, one row per CTA
    [1700, 457, 30, 1],      # two rows in one CTA only
    [4095, 4097, 5],         # eight warps, then nine
    [8192, 153, 3],          # sixteen warps
]


@pytest.mark.parametrize("act", ["tanh", "softplus"])
@pytest.mark.parametrize("case", range(len(SHAPES)))
def test_residual(case, act):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_22462_gb300 import build, nnc
    build.build()
    widths = SHAPES[case]
    rng = np.random.default_rng(case)
    W = [rng.standard_normal((m, k)) / np.sqrt(k) for k, m in zip(widths, widths[1:])]
    b = [0.1 * rng.standard_normal(m) for m in widths[1:]]
    x, y = rng.random(widths[0]), rng.standard_normal(widths[-1])
    net = nnc.Net(widths, [act] * (len(W) - 1) + ["identity"], W, b, "fp32")
    r, v = net.residual(x, y), net.eval(x)
    a = x
    for l, w in enumerate(W):
        a = w @ a + b[l]
        if l + 1 < len(W):
            a = np.tanh(a) if act == "tanh" else np.logaddexp(0.0, a)
    net.free()
    tol = 1e-10 * max(1.0, np.abs(a).max())
    assert np.abs(r - (y - a)).max() < tol
    assert np.abs(v - a).max() < tol


def test_batch_of_many_rows_per_cta():
    """57 networks of 1664-wide layers: 104 rows per CTA of four warps and the finishing one, so that the two
    buffers of partial sums are used again."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_22462_gb300 import build, nnc
    build.build()
    rng = np.random.default_rng(0)
    widths = [20, 1664, 1664, 1]
    W = [rng.standard_normal((m, k)) / np.sqrt(k) for k, m in zip(widths, widths[1:])]
    b = [0.1 * rng.standard_normal(m) for m in widths[1:]]
    nets = [nnc.Net(widths, ["tanh", "tanh", "identity"], W, b, "bf16") for _ in range(57)]
    batch = nnc.Batch(nets)
    xs = [rng.random(20) for _ in nets]
    ys = [np.zeros(1) for _ in nets]
    want = []
    for x in xs:
        a = x
        for l, w in enumerate(W):
            a = w @ a + b[l]
            a = np.tanh(a) if l < 2 else a
        want.append(a)
    got = [np.asarray(r) for r in batch.residual(xs, ys)]
    batch.free()
    for n in nets:
        n.free()
    assert max(np.abs(g + a).max() for g, a in zip(got, want)) < 1e-10
