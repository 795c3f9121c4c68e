"""GPU: calls of the gated layer that leave the usual route, against float64 on the CPU."""
import pytest

from gpu_common import normwise

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def float64(layer, h):
    """The layer and its input in float64 on the CPU, and its output by its modules
    one by one, the scan step by step."""
    import copy
    m = copy.deepcopy(layer).cpu().double()
    h = h.detach().double().cpu().requires_grad_()
    hx, hz = m.in_proj(h).chunk(2, dim=-1)
    x = torch.nn.functional.silu(m.conv(hx.transpose(1, 2))[..., :h.shape[1]].transpose(1, 2))
    r, i = torch.sigmoid(m.gate_proj(x)).chunk(2, dim=-1)
    a = torch.exp(-m.c * torch.nn.functional.softplus(m.lam) * r)
    u, state, ys = torch.sqrt(1 - a * a) * i * x, 0.0, []
    for t in range(h.shape[1]):
        state = a[:, t] * state + u[:, t]
        ys.append(state)
    return m, h, m.out_proj(torch.stack(ys, 1) * torch.nn.functional.silu(hz))


def close(got, want, tol):
    assert normwise(got.detach().double().cpu().numpy(), want.detach().numpy()) <= tol


@pytest.mark.parametrize("kw", [dict(padding=6, dilation=2), dict(padding=3, padding_mode="circular")])
def test_other_convolutions(kw):
    from paper_2406_12580_gb300.layer import GatedRecurrentLayer
    torch.manual_seed(11)
    layer = GatedRecurrentLayer(16, device="cuda")
    layer.conv = torch.nn.Conv1d(32, 32, 4, groups=32, device="cuda", **kw)
    h = torch.randn(2, 21, 16, device="cuda")
    with torch.backends.cudnn.flags(enabled=True, allow_tf32=False):
        got = layer(h)
    # float32 throughout: the bound of the layer's kernels (1e-5)
    close(got, float64(layer, h)[2], 1e-5)


def test_gradients_of_gradients():
    """A gradient penalty of the whole layer, scan included. Float32 evaluations of
    the formulas over 20 steps whose 1 / (1 - alpha^2) is about 10: 2^-24 * 20 * 10
    * 10 operations, 1e-4."""
    from paper_2406_12580_gb300.layer import GatedRecurrentLayer
    torch.manual_seed(12)
    layer = GatedRecurrentLayer(16, device="cuda")
    h = torch.randn(3, 20, 16, device="cuda", requires_grad=True)
    y = layer(h)
    assert "LayerF32" in type(y.grad_fn).__name__
    m, h64, y64 = float64(layer, h)
    both = []
    for mod, inp, out in ((layer, h, y), (m, h64, y64)):
        ins = [inp, *mod.parameters()]
        first = torch.autograd.grad(out.square().sum(), ins, create_graph=True)
        both.append(first + torch.autograd.grad(sum(g.square().sum() for g in first), ins))
    for got, want in zip(*both):
        close(got, want, 1e-4)


@pytest.mark.parametrize("how", ["eager", "captured", "captured at once"])
@pytest.mark.parametrize("B,L", [(2, 20), (35, 20), (33, 31), (60, 31)])
def test_projections_by_either_product(monkeypatch, B, L, how):
    """Captured after an eager pass, one, two or all of the layer's projections (128 x 32, 128 x 64, 32 x
    64) run on the library's kernels and the others on torch's products, by the rows;
    else all on the kernels: the output and every gradient. Five float32 stages of 1e-5 each."""
    import threading

    from paper_2406_12580_gb300 import layer as layer_module
    from paper_2406_12580_gb300.layer import GatedRecurrentLayer, _own_product
    monkeypatch.setattr(layer_module, "_products", threading.local())
    torch.manual_seed(13)
    layer = GatedRecurrentLayer(32, device="cuda")
    h = torch.randn(B, L, 32, device="cuda", requires_grad=True)
    dy = torch.randn(B, L, 32, device="cuda")

    def run():
        y = layer(h)
        assert "LayerF32" in type(y.grad_fn).__name__
        own = [_own_product(B * L, n, k) for n, k in ((128, 32), (128, 64), (32, 64))]
        assert own == ([B * L >= 640, B * L >= 906, True] if how == "captured" else [True] * 3)
        return y, *torch.autograd.grad(y, [h, *layer.parameters()], dy)

    if how == "captured":
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            layer(h).backward(dy)  # a capture follows an eager pass
        torch.cuda.current_stream().wait_stream(side)
    if how != "eager":
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            got = run()
        graph.replay()
    else:
        got = run()
    m, h64, y64 = float64(layer, h)
    want = torch.autograd.grad(y64, [h64, *m.parameters()], dy.double().cpu())
    for g, w in zip(got, (y64, *want)):
        close(g, w, 5e-5)


def test_nans_stay_in_their_rows():
    """A NaN in one sequence reaches its later steps, and gradients of the weights, but
    no other sequence (the layer's kernels, at tails of their tiles)."""
    from paper_2406_12580_gb300.layer import GatedRecurrentLayer
    torch.manual_seed(14)
    layer = GatedRecurrentLayer(12, device="cuda")
    h = torch.randn(5, 37, 12, device="cuda")
    h[2, 20, 3] = float("nan")
    h.requires_grad_()
    dy = torch.randn(5, 37, 12, device="cuda")
    y = layer(h)
    assert "LayerF32" in type(y.grad_fn).__name__
    dh, dw = torch.autograd.grad(y, [h, layer.in_proj.weight], dy)
    m, h64, y64 = float64(layer, h)
    dh64, dw64 = torch.autograd.grad(y64, [h64, m.in_proj.weight], dy.double().cpu())
    for got, want in ((y, y64), (dh, dh64), (dw, dw64)):
        nan = torch.isnan(want)
        assert nan.any() and torch.equal(torch.isnan(got).cpu(), nan)
        if not nan.all():
            close(got.detach()[~nan.cuda()], want[~nan], 5e-5)


def test_compiled_layer():
    """torch.compile breaks its graph at the scan and goes on: the eager layer's output
    and gradients, from torch's operators around the scan (1e-5 as any of them)."""
    from paper_2406_12580_gb300.layer import GatedRecurrentLayer
    torch.manual_seed(15)
    layer = GatedRecurrentLayer(16, device="cuda")
    h = torch.randn(3, 40, 16, device="cuda", requires_grad=True)
    both = []
    for call in (layer, torch.compile(layer, backend="eager")):
        y = call(h)
        both.append((y, *torch.autograd.grad(y.square().sum(), [h, *layer.parameters()])))
    for got, want in zip(*reversed(both)):
        close(got, want.cpu(), 1e-5)
