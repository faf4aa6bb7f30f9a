"""The FP32 GEMM behind the plain MLPs (and the FP32 network) at tile edges: odd widths and row
counts, rows on 4-, 8- and 16-byte boundaries, one-column and one-row outputs, inner sizes
below and above the split threshold, tuned and untuned.  Weights, inputs and gradients are
positive, so every sum has positive terms and each result's relative error is at most the
number of its roundings (the inner sizes it passed through, a few per layer more) times
2^-24, against FP64 torch autograd."""
import numpy as np
import pytest

from paper_1709_05418_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def reference(widths, params, x, dout):
    p = params.double().requires_grad_(True)
    h, prev, off = x.double(), x.shape[1], 0
    for w in list(widths) + [1]:
        h = torch.relu(h @ p[off:off + w * prev].reshape(w, prev).t() + p[off + w * prev:off + w * prev + w])
        off += w * prev + w
        prev = w
    (h[:, 0] * dout.double()).sum().backward()
    return h[:, 0].detach(), p.grad


@pytest.mark.parametrize("tuned", [False, True])
@pytest.mark.parametrize("widths,din", [((200, 200), 226), ((1, 33, 130), 51), ((64, 7), 2400), ((257,), 18)])
@pytest.mark.parametrize("q", [1, 63, 65, 129, 1100])
def test_dense_at_tile_edges(widths, din, q, tuned):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1709_05418_gb300 import api
    ctx = api.Context()
    ctx.set_autotune(tuned)
    g = torch.Generator().manual_seed(q + din)
    params = torch.from_numpy(np.abs(W.dense_he_init(widths, din, seed=3, bias=0.1))).cuda()
    x = (torch.rand((q, din), generator=g) + 0.1).cuda()
    dout = (torch.rand(q, generator=g) + 0.1).cuda()
    out, grad = reference(widths, params, x, dout)
    inner = [din] + list(widths)
    fwd = (sum(inner) + 4 * len(inner)) * 2.0 ** -24
    bwd = (2 * sum(inner) + q + 8 * len(inner)) * 2.0 ** -24
    got = ctx.dense_forward(widths, params, x).double()
    assert float(((got - out).abs() / out).max()) <= fwd
    got = ctx.dense_backward(widths, params, x, dout).double()
    assert float(((got - grad).abs() / grad).max()) <= bwd
    ctx.close()


def test_tuned_rows_beyond_the_low_tiles():
    """2,097,121 rows, one more than 65,535 tiles of 32 hold: tuned calls and calls with a 32-row tile
    from a table run (they are accepted up to 65,535 x 64) and give the default tile's bits."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1709_05418_gb300 import api
    q, widths, din = 32 * 65535 + 1, (8,), 4
    params = torch.from_numpy(W.dense_he_init(widths, din, seed=3, bias=0.1)).cuda()
    x = torch.rand((q, din), generator=torch.Generator().manual_seed(1)).cuda()
    tuned, plain, given = api.Context(), api.Context(), api.Context()
    plain.set_autotune(False)
    ref = plain.dense_forward(widths, params, x)
    assert torch.equal(tuned.dense_forward(widths, params, x), ref)
    given.set_autotune_table([dict(e, tile_m=32, tile_n=64, tile_k=16) for e in tuned.autotune_table()])
    assert torch.equal(given.dense_forward(widths, params, x), ref)
    for c in (tuned, plain, given):
        c.close()


def small_terms(n):
    """1, then n - 1 terms of 2^-25: added to 1 one by one, each is rounded away."""
    t = torch.full((n,), 2.0 ** -25)
    t[0] = 1.0
    return t


@pytest.mark.parametrize("K,q", [(2400, 1), (2400, 130), (4096, 65), (16384, 3)])
def test_long_one_column_sums_keep_their_terms(K, q):
    """No hidden layer: output = a sum of K products.  In runs of at most K / 16 terms (the tuner's
    fewest above 1,024) the first run loses K / 16 of the small terms at the most, 2^-25 each; a
    chain of all of them loses K - 1.  Also the last layer of a K-wide network, from relu(x w) = w."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1709_05418_gb300 import api
    ctx = api.Context()
    terms = small_terms(K).cuda()
    exact = float(terms.double().sum())
    bound = (K / 16) * 2.0 ** -25 + 64 * 2.0 ** -24        # and one rounding per run, two runs' worth
    params = torch.cat([terms, torch.zeros(1, device="cuda")])
    got = ctx.dense_forward((), params, torch.ones((q, K), device="cuda"))
    assert float((got.double() - exact).abs().max()) <= bound
    wide = torch.cat([torch.ones(K, device="cuda"), torch.zeros(K, device="cuda"), params])
    got = ctx.dense_forward((K,), wide, torch.ones((q, 1), device="cuda"))
    assert float((got.double() - exact).abs().max()) <= bound
    ctx.close()


def test_long_sums_over_rows_of_one_wide_layers_keep_their_terms():
    """The weight gradient of a 1-wide layer on 1 input is one sum over the rows."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1709_05418_gb300 import api
    ctx = api.Context()
    q = 16384
    dout = small_terms(q).cuda()
    params = torch.tensor([1.0, 0.0, 1.0, 0.0], device="cuda")          # w, b, w_out, b_out
    grad = ctx.dense_backward((1,), params, torch.ones((q, 1), device="cuda"), dout).double()
    exact = float(dout.double().sum())
    assert abs(float(grad[0]) - exact) <= (q / 16) * 2.0 ** -25 + 64 * 2.0 ** -24
    ctx.close()


def test_grouped_gradients_do_not_share_a_plain_gradients_tile():
    """The network's 31 weight gradients are one launch and a 200 x 200 plain layer's is one GEMM:
    each is timed by itself, so neither's split nor speed depends on which ran first.  Networks of
    another input width group other problems."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1709_05418_gb300 import api
    q = 64
    g = torch.Generator().manual_seed(8)
    ctx = api.Context()

    def entries():
        return {(e["M"], e["N"], e["K0"], e["K1"], e["flags"]) for e in ctx.autotune_table() if e["K0"] == q}

    params = torch.from_numpy(W.dense_he_init((200, 200), 200, seed=3, bias=0.1)).cuda()
    ctx.dense_backward((200, 200), params, torch.rand((q, 200), generator=g).cuda(), torch.rand(q, generator=g).cuda())
    plain = entries()
    assert plain
    for n_xy, din in ((5, 226), (2, 13)):
        before = entries()
        n = ctx.stencil_param_count(n_xy)
        ctx.stencil_backward(n_xy, torch.randn(n, generator=g).cuda() * 0.05, torch.rand((q, 10, din), generator=g).cuda(),
                             torch.rand(q, generator=g).cuda())
        new = [k for k in entries() - before if k[0] == 200]
        assert len(new) == 1 and new[0][:4] == (200, max(din, 200), q, 31), new
    ctx.close()
