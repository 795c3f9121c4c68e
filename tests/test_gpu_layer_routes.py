"""GPU: calls of the gated layer that leave the usual route, against float64 on the CPU."""
import pytest

from gpu_common import normwise

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def reference(layer, h):
    """The layer's output in float64, its modules called one by one, the scan step by step."""
    import copy
    m = copy.deepcopy(layer).cpu().double()
    h, L = h.detach().double().cpu(), h.shape[1]
    hx, hz = m.in_proj(h).chunk(2, dim=-1)
    x = torch.nn.functional.silu(m.conv(hx.transpose(1, 2))[..., :L].transpose(1, 2))
    r, i = torch.sigmoid(m.gate_proj(x)).chunk(2, dim=-1)
    a = torch.exp(-m.c * torch.nn.functional.softplus(m.lam) * r)
    u, state, ys = torch.sqrt(1 - a * a) * i * x, 0.0, []
    for t in range(L):
        state = a[:, t] * state + u[:, t]
        ys.append(state)
    return m.out_proj(torch.stack(ys, 1) * torch.nn.functional.silu(hz)).detach().numpy()


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
    assert normwise(got.detach().cpu().numpy(), reference(layer, h)) <= 1e-5
