"""CPU: which calls of the gated layer may take the library's kernels."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
from torch import nn  # noqa: E402

from paper_2406_12580_gb300 import layer as layer_module  # noqa: E402


def test_the_convolutions_settings_are_honoured():
    """A convolution with other settings than the kernels' is called as a module."""
    layer = layer_module.GatedRecurrentLayer(8)
    assert layer._conv_ok()
    for kw in (dict(padding=6, dilation=2), dict(padding=3, padding_mode="circular"),
               dict(padding=3, padding_mode="reflect"), dict(padding=3, stride=2),
               dict(padding=0), dict(padding="same")):
        layer.conv = nn.Conv1d(16, 16, 4, groups=16, **kw)
        assert not layer._conv_ok(), kw


def test_a_hook_on_every_module_sees_the_convolution():
    layer, seen = layer_module.GatedRecurrentLayer(8), []
    hook = nn.modules.module.register_module_forward_hook(lambda m, i, o: seen.append(type(m)))
    try:
        assert not layer._conv_ok()
        layer._conv_silu(torch.randn(2, 5, 32))
    finally:
        hook.remove()
    assert seen == [nn.Conv1d] and layer._conv_ok()


ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("setting,tf32", [
    ("torch.backends.cuda.matmul.fp32_precision = 'tf32'", True),
    ("torch.backends.fp32_precision = 'tf32'", True),
    ("torch.backends.cuda.matmul.fp32_precision = 'ieee'", False),
    ("torch.backends.cuda.matmul.allow_tf32 = True", True),
    ("torch.set_float32_matmul_precision('high')", True), ("pass", False)])
def test_tf32_by_either_setting(setting, tf32):
    """TF32 allowed by the older or the newer setting leaves float32 projections
    with torch, and neither makes the call raise. (A process of its own: the
    settings are the process's.)"""
    if "fp32_precision" in setting and not hasattr(torch.backends.cuda.matmul, "fp32_precision"):
        pytest.skip("no such setting in this torch")
    code = f"""
import torch
from paper_2406_12580_gb300 import layer as m
{setting}
lin, x = m._Linear(8, 8), torch.randn(3, 8)
layer, h = m.GatedRecurrentLayer(8), torch.randn(2, 3, 8)
lin(x)
m._plain_cuda = lambda *a: True
class Kernel:
    apply = staticmethod(lambda x, w, b: "kernel")
m._LinearF32 = Kernel
assert isinstance(lin(x), str) != {tf32}
assert (layer._whole(h) is None) == {tf32}
"""
    subprocess.run([sys.executable, "-W", "ignore", "-c", code], check=True, cwd=ROOT)


@pytest.fixture
def kernels_on_cpu(monkeypatch):
    """Stands torch operators in for the library's calls, out of autograd's sight as those are."""
    def linear_fwd(T, N, K, x, w, b, y):
        assert x.is_contiguous() and w.is_contiguous()
        y.copy_(nn.functional.linear(x, w, b))

    def conv_fwd(B, L, C, io, hxz, w, b, x, z):
        assert hxz.is_contiguous()
        for to, of in zip((x, z), layer_module._conv_silu_torch(hxz.view(B, L, 2 * C), w, b)):
            to.copy_(of.reshape(to.shape))

    def definition(c, x, gl, lam, z, h0):
        """The gated scan in float64, written out from Sec. 3.2."""
        D = x.shape[2]
        r, i = torch.sigmoid(gl[..., :D]), torch.sigmoid(gl[..., D:])
        a = torch.exp(-c * r * torch.log1p(torch.exp(lam)))
        h, hs = (0.0 if h0 is None else h0), []
        for t in range(x.shape[1]):
            h = a[:, t] * h + torch.sqrt(1 - a[:, t] ** 2) * i[:, t] * x[:, t]
            hs.append(h)
        return torch.stack(hs, 1) * z * torch.sigmoid(z), h

    def scan_fwd(desc, x, gl, lam, h0, z, y, h_last, ws):
        ins = [t.double().view(desc.B, desc.L, -1) for t in (x, gl, z)]
        ins = (ins[0], ins[1], lam.double(), ins[2], None if h0 is None else h0.double())
        for to, of in zip((y, h_last), definition(desc.c, *ins)):
            if to is not None:
                to.copy_(of.reshape(to.shape))

    def scan_bwd(desc, dy, dh_last, x, gl, lam, h0, z, dx, dgl, dz, dlam, dh0, ws):
        with torch.enable_grad():
            ins = [None if t is None else t.detach().double().requires_grad_() for t in (x, gl, lam, z, h0)]
            outs = definition(desc.c, *ins)
            dh_last = torch.zeros_like(outs[1]) if dh_last is None else dh_last
            got = torch.autograd.grad(outs, [t for t in ins if t is not None],
                                      (dy.double(), dh_last.double()))
        for to, of in zip((dx, dgl, dlam, dz, dh0), got):
            to.copy_(of)

    monkeypatch.setattr(layer_module, "blr_scan_fwd_gated", scan_fwd)
    monkeypatch.setattr(layer_module, "blr_scan_bwd_gated", scan_bwd)
    monkeypatch.setattr(layer_module, "blr_workspace_bytes", lambda d: 64)
    monkeypatch.setattr(layer_module, "_dtype_code", lambda t: 0)
    monkeypatch.setattr(layer_module, "_own_products", lambda T, sizes, forward: (True,) * len(sizes))
    kernels = dict(definition=definition)
    monkeypatch.setattr(layer_module, "blr_linear_fwd", linear_fwd)
    monkeypatch.setattr(layer_module, "blr_conv_silu_fwd", conv_fwd)
    return kernels


def _grads(out, inputs, create_graph):
    """First gradients of a scalar and, with create_graph, those of their squares."""
    first = torch.autograd.grad(out, inputs, create_graph=create_graph)
    if not create_graph:
        return first
    return first + torch.autograd.grad(sum(g.square().sum() for g in first), inputs)


@pytest.mark.parametrize("graph", [True, False])
def test_gradients_by_torch_operators_are_this_calls_own(kernels_on_cpu, graph):
    """Where a backward uses torch operators (create_graph; gradients the kernels
    do not take), its gradients are those of its own call: of a projection or a
    convolution applied twice, whose second input depends on the same weights, and
    of inputs that are views of other strides."""
    torch.manual_seed(5)
    rand = lambda *s: torch.randn(*s, dtype=torch.float64, requires_grad=True)  # noqa: E731
    w, b, x = rand(6, 6), rand(6), rand(6, 5)
    k, c, h = rand(4, 1, 4), rand(4), rand(8, 7, 2)
    lin, conv = layer_module._LinearF32.apply, layer_module._ConvSiLU.apply
    for lin_, conv_ in ((lin, conv), (nn.functional.linear, layer_module._conv_silu_torch)):
        y = lin_(lin_(x.t(), w.t(), b), w.t(), b)
        once = torch.cat(conv_(h.transpose(0, 2), k, c), dim=-1)
        z, _ = conv_(once, k, c)
        got = _grads(y.square().sum(), (x, w, b), graph) + _grads(z.square().sum(), (h, k, c), graph)
        if lin_ is lin:
            kernel = got
    for a, r in zip(kernel, got):  # the same operators in the same precision: float64's rounding
        assert (a - r).abs().max() <= 1e-12 * r.abs().max() and a.requires_grad == r.requires_grad


@pytest.mark.parametrize("state", [False, True])
def test_second_gradients_pass_through_the_scan(kernels_on_cpu, state):
    """A gradient penalty through the gated scan has every term, for inputs of other
    strides too, and the first gradients under create_graph are the kernels'. Both
    sides are float32 evaluations of the same formulas over 12 steps whose 1 / (1 -
    alpha^2) is about 10: 2^-24 * 12 * 10 * 10 operations, 1e-4."""
    torch.manual_seed(9)
    rand = lambda *s: torch.randn(*s, requires_grad=True)  # noqa: E731
    x, gl, lam, z = rand(6, 12, 3), rand(3, 12, 12), rand(6), rand(3, 12, 6)
    h0 = rand(3, 6) if state else None
    ins = [t for t in (x, gl, lam, z, h0) if t is not None]
    seen = []
    for scan, to in ((layer_module.BDLRUGatedScan.apply, torch.Tensor.float),
                     (lambda x, gl, lam, z, h0: kernels_on_cpu["definition"](1.0, x, gl, lam, z, h0),
                      torch.Tensor.double)):
        args = [None if t is None else to(t) for t in (x.transpose(0, 2), gl, lam, z, h0)]
        y, h_last = scan(*args)
        seen.append(_grads((y.square().sum() + h_last.sum()).sum(), ins, True))
    for a, r in zip(*seen):
        assert (a - r).abs().max() <= 1e-4 * r.abs().max()


def test_second_gradients_of_the_whole_layer(kernels_on_cpu, monkeypatch):
    torch.manual_seed(10)
    layer, h = layer_module.GatedRecurrentLayer(8), torch.randn(2, 9, 8, requires_grad=True)
    p = [dict(layer.named_parameters())[n] for n in
         ("in_proj.weight", "in_proj.bias", "conv.weight", "conv.bias", "gate_proj.weight",
          "gate_proj.bias", "lam", "out_proj.weight", "out_proj.bias")]
    out = layer_module._LayerF32.apply(1.0, h, *p)
    got = _grads(out.square().sum(), [h, *p], True)
    p64, h64 = [t.detach().double().requires_grad_() for t in p], h.detach().double().requires_grad_()
    hxz = nn.functional.linear(h64, p64[0], p64[1])
    x, z = layer_module._conv_silu_torch(hxz, p64[2], p64[3])
    y, _ = kernels_on_cpu["definition"](1.0, x, nn.functional.linear(x, p64[4], p64[5]), p64[6], z, None)
    want = _grads(nn.functional.linear(y, p64[7], p64[8]).square().sum(), [h64, *p64], True)
    for a, r in zip(got, want):
        assert (a - r).abs().max() <= 1e-4 * r.abs().max()


@pytest.fixture
def device_state(monkeypatch):
    """The calls by which the rule for a projection asks about the device."""
    state = dict(capturing=False, handles=0)
    monkeypatch.setattr(torch._C, "_cuda_getDevice", lambda: 0, raising=False)
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: state["capturing"])
    monkeypatch.setattr(torch.cuda, "current_blas_handle",
                        lambda: state.update(handles=state["handles"] + 1))
    monkeypatch.setattr(layer_module, "_products", type(layer_module._products)())
    return state


def test_rule_for_a_projection(device_state):
    """The library's kernels where they are the faster, or launched the faster; in a
    capture by device time, but torch's products only once they have been set up in
    the thread, by an eager pass."""
    own, state = layer_module._own_product, device_state
    always = ((50, 64, 32), (51200, 256, 128), (10240, 1024, 256))
    eager = ((50, 256, 128), (200, 1024, 512), (4000, 1024, 256))
    never = ((200, 2048, 1024), (51200, 1024, 1024), (3000, 1024, 512))
    state["capturing"] = True
    assert all(own(*s) for s in always + eager + never)
    state["capturing"] = False
    assert all(own(*s) for s in always) and state["handles"] == 0
    assert all(own(*s) for s in eager) and state["handles"] == 1
    assert not any(own(*s) for s in never)
    state["capturing"] = True
    assert all(own(*s) for s in always) and not any(own(*s) for s in eager + never)
    assert state["handles"] == 1
    assert not own(50, 65540, 4) and not own(50, 6, 4)  # the kernels refuse them
    assert own(51200, 2048, 512, True) and not own(51200, 2048, 512, False)
    assert not own(1600, 1024, 512, True) and not own(51200, 2048, 1024, True)


@pytest.mark.parametrize("n,k,kernel", [(65536, 4, True), (65540, 4, False), (4, 65540, False),
                                        (6, 4, False), (4, 6, False)])
def test_projections_the_kernels_refuse_stay_with_torch(monkeypatch, device_state, n, k, kernel):
    monkeypatch.setattr(layer_module, "_plain_cuda", lambda *a: True)
    called = []
    monkeypatch.setattr(layer_module, "blr_linear_fwd", lambda *a: called.append(a))
    y = layer_module._Linear(k, n)(torch.randn(2, k))
    assert y.shape == (2, n) and len(called) == kernel


@pytest.mark.parametrize("name,shape", [
    ("in_proj.weight", (40, 8)), ("in_proj.bias", (16,)), ("conv.bias", (8,)),
    ("gate_proj.weight", (32, 8)), ("gate_proj.bias", (16,)), ("lam", (8,)),
    ("out_proj.weight", (8, 32)), ("out_proj.bias", (4,)), ("in_proj.weight", (48, 8))])
def test_parameters_of_other_sizes_never_reach_the_kernels(monkeypatch, name, shape):
    """The kernels read as many values as the sizes say: a parameter of another size
    goes to the operators one by one, which refuse it."""
    layer, h = layer_module.GatedRecurrentLayer(8), torch.randn(2, 5, 8)
    monkeypatch.setattr(layer_module, "_plain_cuda", lambda *a: True)
    assert layer._whole(h) is not None
    module, _, attr = name.rpartition(".")
    setattr(layer.get_submodule(module), attr, nn.Parameter(torch.randn(shape)))
    assert layer._whole(h) is None
    refuse = lambda *a: pytest.fail("a kernel was called")  # noqa: E731
    if module == "conv":
        monkeypatch.setattr(layer_module._ConvSiLU, "apply", staticmethod(refuse))
        with pytest.raises(RuntimeError):
            layer._conv_silu(torch.randn(2, 5, 32))
    elif name == "in_proj.weight":
        monkeypatch.setattr(layer_module._ConvSiLU, "apply", staticmethod(refuse))
        with pytest.raises((RuntimeError, ValueError)):
            layer._conv_silu(torch.randn(2, 5, shape[0]))
    elif name == "lam":
        x = torch.randn(2, 5, 16)
        with pytest.raises(ValueError, match="lam: fewer values"):
            layer_module.BDLRUGatedScan.apply(x, torch.randn(2, 5, 32), layer.lam, x)
    else:
        monkeypatch.setattr(layer_module._LinearF32, "apply", staticmethod(refuse))
        lin = getattr(layer, module)
        with pytest.raises(RuntimeError):
            lin(torch.randn(3, 16 if module != "in_proj" else 8))


def test_saved_tensors_are_unpacked_once(kernels_on_cpu):
    """Hooks that bring a saved tensor back (from another memory, say) run once a backward."""
    rand = lambda *s: torch.randn(*s, requires_grad=True)  # noqa: E731
    packed, unpacked = [], []
    with torch.autograd.graph.saved_tensors_hooks(lambda t: packed.append(t.shape) or t,
                                                  lambda t: unpacked.append(t.shape) or t):
        y, _ = layer_module.BDLRUGatedScan.apply(rand(2, 3, 8), rand(2, 3, 16), rand(8), rand(2, 3, 8),
                                                 rand(2, 8))
    y.backward(torch.ones_like(y))
    assert len(packed) == len(unpacked) == 6
