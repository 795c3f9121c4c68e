"""GPU: the gated layer's convolution and projection kernels against the same
operators in float64 on the CPU.

Bounds (normwise): a float32 output of K multiply-adds in float32 stays within
K 2^-24 of the sum of its terms' magnitudes, and the normwise error is against
the largest output, which is of the order of sqrt(K) of the terms; 1e-5 covers
the sums here (K up to 300 forward, and 5000 in the weight gradients, which are
summed in parts). bfloat16 outputs are rounded once, 2^-8."""
import pytest

from gpu_common import normwise

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def _close(got, want, tol, name):
    assert got.dtype != torch.float64 and got.shape == want.shape, name
    assert normwise(got.detach().double().cpu().numpy(), want.detach().cpu().numpy()) <= tol, name


# rows, outputs, inputs: single tiles, their edges, more than one tile and split
@pytest.mark.parametrize("T,N,K", [(1, 4, 4), (15, 64, 16), (128, 128, 64), (129, 132, 68),
                                   (300, 20, 300), (5000, 256, 128), (2049, 512, 8)])
def test_linear(T, N, K):
    from paper_2406_12580_gb300.layer import _Linear, _LinearF32
    torch.manual_seed(T + N + K)
    lin = _Linear(K, N, device="cuda")
    x = torch.randn(T, K, device="cuda", requires_grad=True)
    dy = torch.randn(T, N, device="cuda")
    y = lin(x)
    assert type(y.grad_fn).__name__ == _LinearF32.__name__ + "Backward"
    got = torch.autograd.grad(y, [x, lin.weight, lin.bias], dy)
    x64, w64, b64 = (t.detach().double().cpu().requires_grad_() for t in (x, lin.weight, lin.bias))
    y64 = torch.nn.functional.linear(x64, w64, b64)
    want = torch.autograd.grad(y64, [x64, w64, b64], dy.double().cpu())
    _close(y, y64, 1e-5, "y")
    for g, w, name in zip(got, want, ("dx", "dw", "db")):
        _close(g, w, 1e-5, name)


# one row, the taps' edges, a chunk of rows and its edges, several blocks
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("B,L,C", [(1, 1, 8), (2, 3, 8), (3, 32, 24), (2, 33, 136), (5, 100, 64),
                                   (40, 67, 128), (2, 40, 1024)])
def test_conv_silu(B, L, C, dtype):
    from paper_2406_12580_gb300.layer import _ConvSiLU, _conv_silu_torch
    torch.manual_seed(B + L + C)
    mk = lambda *s: torch.randn(*s, device="cuda").to(dtype).requires_grad_()  # noqa: E731
    hxz, w, b = mk(B, L, 2 * C), mk(C, 1, 4), mk(C)
    dx, dz = mk(B, L, C).detach(), mk(B, L, C).detach()
    outs = _ConvSiLU.apply(hxz, w, b)
    got = torch.autograd.grad(outs, [hxz, w, b], (dx, dz))
    in64 = [t.detach().double().cpu().requires_grad_() for t in (hxz, w, b)]
    outs64 = _conv_silu_torch(*in64)
    want = torch.autograd.grad(outs64, in64, (dx.double().cpu(), dz.double().cpu()))
    tol = 1e-5 if dtype == torch.float32 else 2.0 ** -8
    for g, wv, name in zip((*outs, *got), (*outs64, *want), ("x", "z", "dhxz", "dw", "db")):
        _close(g, wv, tol, name)


def test_layer_keeps_torch_where_it_must():
    """Autocast, TF32 and a hook on the convolution run the torch operators;
    second derivatives of the projections and the convolution stay available."""
    from paper_2406_12580_gb300.layer import (GatedRecurrentLayer, _ConvSiLU, _conv_silu_torch,
                                              _LinearF32)
    torch.manual_seed(3)
    layer = GatedRecurrentLayer(16, device="cuda")
    h = torch.randn(3, 20, 16, device="cuda")
    want = layer(h)
    assert "LayerF32" in type(want.grad_fn).__name__
    with torch.autocast("cuda", dtype=torch.bfloat16):
        assert layer.in_proj(h).dtype == torch.bfloat16
    torch.backends.cuda.matmul.allow_tf32 = True
    try:
        assert "LinearF32" not in type(layer.in_proj(h).grad_fn).__name__
    finally:
        torch.backends.cuda.matmul.allow_tf32 = False
    seen = []
    layer.conv.register_forward_hook(lambda m, i, o: seen.append(o.shape))
    assert normwise(layer(h).detach().cpu().numpy(), want.detach().cpu().numpy()) <= 1e-5 and seen
    x, w, b = (torch.randn(*s, device="cuda", requires_grad=True) for s in ((5, 8), (12, 8), (12,)))
    dx, = torch.autograd.grad(_LinearF32.apply(x, w, b).square().sum(), x, create_graph=True)
    ddw, = torch.autograd.grad(dx.sum(), w)
    rx, = torch.autograd.grad(torch.nn.functional.linear(x, w, b).square().sum(), x, create_graph=True)
    rdw, = torch.autograd.grad(rx.sum(), w)
    assert normwise(ddw.cpu().numpy(), rdw.cpu().numpy()) <= 1e-5
    c = [torch.randn(*s, device="cuda", requires_grad=True) for s in ((2, 9, 16), (8, 1, 4), (8,))]
    two = []
    for fn in (_ConvSiLU.apply, _conv_silu_torch):
        g, = torch.autograd.grad(fn(*c)[0].square().sum(), c[0], create_graph=True)
        two.append(torch.autograd.grad(g.square().sum(), c[1])[0])
    assert normwise(two[0].cpu().numpy(), two[1].cpu().numpy()) <= 1e-4


def test_modes_and_tracing_see_torch_operators():
    """A dispatch or function mode and torch.jit.trace get the projections and the
    convolution as torch operators; a negative view is read as the values it has."""
    from torch.overrides import TorchFunctionMode
    from torch.utils._python_dispatch import TorchDispatchMode

    from paper_2406_12580_gb300.layer import GatedRecurrentLayer, _Linear
    seen = []

    class Dispatch(TorchDispatchMode):
        def __torch_dispatch__(self, func, types, args=(), kwargs=None):
            seen.append(str(func))
            return func(*args, **(kwargs or {}))

    class Function(TorchFunctionMode):
        def __torch_function__(self, func, types, args=(), kwargs=None):
            seen.append(getattr(func, "__name__", ""))
            return func(*args, **(kwargs or {}))

    torch.manual_seed(7)
    layer = GatedRecurrentLayer(16, device="cuda")
    h = torch.randn(2, 12, 16, device="cuda")
    want = layer(h)
    for mode, ops in ((Dispatch, ("mm", "conv")), (Function, ("linear", "conv1d"))):
        seen.clear()
        with mode():
            got = layer(h)
        assert all(any(op in s for s in seen) for op in ops), (mode, seen)
        assert normwise(got.detach().cpu().numpy(), want.detach().cpu().numpy()) <= 1e-5
    with torch.device("cuda"):
        assert "LayerF32" in type(layer(h).grad_fn).__name__
    lin = _Linear(16, 8, device="cuda")
    graph = str(torch.jit.trace(lin, h).inlined_graph)
    assert "aten::linear" in graph and "PythonOp" not in graph
    neg = torch.randn(5, 16, dtype=torch.complex64, device="cuda").conj().imag
    ref = torch.nn.functional.linear(neg.clone().resolve_neg(), lin.weight, lin.bias)
    assert neg.is_neg() and normwise(lin(neg).detach().cpu().numpy(), ref.detach().cpu().numpy()) <= 1e-5
