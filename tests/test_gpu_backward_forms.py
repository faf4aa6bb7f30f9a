"""The two forms of the FP32 backward, a launch for all weight gradients and a layer's own launches
above 131,072 rows, against FP64 torch autograd.  Parameters and inputs are positive, so every
ReLU is active, every sum has positive terms, and each gradient's relative error is at most the number
of its roundings times 2^-24: the inner sizes of the layers it passed (626 a block, forward and
backward, 401 at the end) and the rows it sums."""
import pytest

from paper_1709_05418_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
H, DIN = W.H, W.DIN


def network(p, z):
    off = 0

    def take(*shape):
        nonlocal off
        n = 1
        for e in shape:
            n *= e
        off += n
        return p[off - n:off].reshape(shape)

    o = None
    for k in range(W.K):
        V = take(H, DIN)
        W1 = take(H, H) if k else None
        b1, W2, b2 = take(H), take(H, H), take(H)
        f = z[:, k, :DIN] @ V.t() + b1
        if k:
            f = f + o @ W1.t()
        f = torch.relu(f) @ W2.t() + b2
        o = torch.relu(f if o is None else f + o)
    for n in (H, H, 1):
        T, b = take(n, H), take(n)
        o = torch.relu(o @ T.t() + b)
    return o[:, 0]


@pytest.mark.parametrize("q,tuned", [(257, True), (131072, True), (131073, True), (131073, False)])
def test_both_forms_against_fp64(q, tuned):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1709_05418_gb300 import api
    g = torch.Generator(device="cuda").manual_seed(q)
    params = torch.from_numpy(W.he_init(seed=6, bias=0.1)).cuda().abs() * 0.1
    z = torch.zeros((q, W.K, 240), device="cuda")
    z[:, :, :DIN] = torch.rand((q, W.K, DIN), generator=g, device="cuda") + 0.1
    dout = torch.rand(q, generator=g, device="cuda") + 0.1
    ctx = api.Context()
    ctx.set_autotune(tuned)
    ctx.set_weights(params)
    got = ctx.mlp_backward(z, dout).double()
    ctx.close()
    p = params.double().requires_grad_(True)
    for a in range(0, q, 16384):
        (network(p, z[a:a + 16384].double()) * dout[a:a + 16384].double()).sum().backward()
    ref = p.grad
    bound = (2 * (10 * 626 + 401 + 8 * 23) + q) * 2.0 ** -24
    live = ref != 0
    assert torch.equal(got[~live], ref[~live])
    assert float(((got - ref).abs()[live] / ref[live]).max()) <= bound
