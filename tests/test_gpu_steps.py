"""GPU: blr_steps at the number of steps where float32 changes its kernel, at batches'
edges and at channel tails, against float64 torch."""
import pytest

from gpu_common import normwise

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("sequence", [False, True])
@pytest.mark.parametrize("io,state", [(0, 0), (0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize("B,K,D,c", [(1, 1, 8, 1.0), (1300, 7, 8, 1.0), (67, 8, 72, 1.0),
                                     (3, 9, 264, 8.0), (1025, 12, 24, 1.0), (70, 33, 520, 1.0)])
def test_steps(B, K, D, c, io, state, sequence):
    """float32: 1e-5 as the scans; bfloat16 2e-2 (an output rounding, tanh.approx)."""
    from paper_2406_12580_gb300 import blr_steps
    types = (torch.float32, torch.bfloat16)
    g = torch.Generator(device="cuda").manual_seed(B + K + D)
    rand = lambda t, *s: torch.randn(*s, device="cuda", generator=g).to(t)  # noqa: E731
    h, x, gl = rand(types[state], B, D), rand(types[io], B, K, D), rand(types[io], B, K, 2 * D)
    lam = rand(torch.float32, D) - 3.0
    seq = torch.empty_like(x) if sequence else None
    ref, want = h.double(), []
    r, i = torch.sigmoid(gl.double()).chunk(2, dim=-1)
    log_a = -c * torch.nn.functional.softplus(lam.double()) * r
    a, u = torch.exp(log_a), torch.sqrt(-torch.expm1(2 * log_a)) * i * x.double()
    for k in range(K):
        ref = a[:, k] * ref + u[:, k]
        want.append(ref)
    blr_steps(B, K, D, io, state, c, h, x, gl, lam, h, seq)  # in place
    tol = 2e-2 if io or state else 1e-5
    assert normwise(h.double().cpu().numpy(), ref.cpu().numpy()) <= tol
    if sequence:
        assert normwise(seq.double().cpu().numpy(), torch.stack(want, 1).cpu().numpy()) <= tol
