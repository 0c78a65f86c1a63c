"""The fused network kernel at the edges of its tiles: rows around 128, more
tiles than SMs (a CTA then takes several), output counts around its 16-column
pieces, every depth; and a training batch of more tiles than SMs against its
parts.

Inference runs the same MMAs in the same order as the layer-by-layer form, so
the two agree bit for bit. The gradient of a batch is the row-weighted mean of
its parts' gradients; the output gradients are rounded to BF16 (2^-9 each,
independent over thousands of rows) after a division by another row count:
2e-3 in the norm, bounded here by 1e-2.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LO, HI = [-20.0, -20.0, 0.0, 280e9], [500.0, 320.0, 10.0, 320e9]


@pytest.fixture(scope="module")
def sbr():
    import paper_2208_10006_gb300 as m
    return m


def queries(B, seed=0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    lo, hi = torch.tensor(LO, device="cuda"), torch.tensor(HI, device="cuda")
    return (lo + torch.rand(B, 4, device="cuda", generator=g) * (hi - lo)).contiguous()


@pytest.mark.parametrize("B", [1, 127, 128, 129, 2 * 152 * 128 + 5])
@pytest.mark.parametrize("n_out", [1, 15, 20, 33, 128])
def test_rows_and_outputs(sbr, B, n_out):
    m = sbr.MLP(n_out, LO, HI, width=256, depth=2, max_batch=B, seed=3, y_shift=np.arange(n_out), y_scale=1 + np.arange(n_out))
    x = queries(B)
    y = torch.full((B * n_out + 64,), 7.0, device="cuda")
    m.predict(x, out=y)   # what lies behind the last output stays as it was
    m.status()
    assert torch.equal(y[: B * n_out].view(B, n_out), m.predict(x, layered=True)) and (y[B * n_out:] == 7.0).all()


@pytest.mark.parametrize("width", [128, 256])
@pytest.mark.parametrize("depth", [1, 2, 3, 5, 8])
def test_widths_and_depths(sbr, width, depth):
    m = sbr.MLP(6, LO, HI, width=width, depth=depth, max_batch=300, seed=5)
    x = queries(300)
    assert torch.equal(m.predict(x), m.predict(x, layered=True))


def test_outputs_at_an_odd_address(sbr):
    # 20 outputs, but the buffer starts 4 bytes past a multiple of 16
    m = sbr.MLP(20, LO, HI, max_batch=200, seed=5)
    x = queries(200)
    y = torch.zeros(200 * 20 + 1, device="cuda")
    m.predict(x, out=y[1:])
    assert torch.equal(y[1:].view(200, 20), m.predict(x))


@pytest.mark.parametrize("width,depth", [(128, 1), (256, 4), (128, 8)])
def test_a_large_batch_has_the_gradient_of_its_parts(sbr, width, depth):
    B, parts, n_out = 160 * 128 + 77, 5, 20
    x = queries(B, 1)
    y = torch.randn(B, n_out, device="cuda", generator=torch.Generator(device="cuda").manual_seed(2))
    y[::7, 3] = float("nan")

    def grad(xs, ys):
        m = sbr.MLP(n_out, LO, HI, width=width, depth=depth, max_batch=len(xs), seed=9, err_channel=19, err_of=0)
        loss = torch.zeros(1, device="cuda")
        m.train_step(xs.contiguous(), ys.contiguous(), loss)
        m.status()
        return m.params(2).double(), float(loss)

    whole, loss = grad(x, y)
    cuts = np.linspace(0, B, parts + 1).astype(int)
    got = [(b - a, *grad(x[a:b], y[a:b])) for a, b in zip(cuts[:-1], cuts[1:])]
    mean = sum(n * g for n, g, _ in got) / B
    assert float((whole - mean).norm() / mean.norm()) < 1e-2
    assert abs(loss - sum(n * l for n, _, l in got) / B) < 1e-4 * loss


def test_a_repeated_step_gives_the_same_bits(sbr):
    x, y = queries(3000, 1), torch.randn(3000, 20, device="cuda")
    runs = []
    for _ in range(2):
        m = sbr.MLP(20, LO, HI, max_batch=3000, seed=9)
        m.train_step(x, y)
        runs.append((m.params(2), m.params(0)))
    assert torch.equal(runs[0][0], runs[1][0]) and torch.equal(runs[0][1], runs[1][1])
