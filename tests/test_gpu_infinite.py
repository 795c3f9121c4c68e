"""GPU: infinite values pass through the scans as through the definition (alpha inf =
inf for alpha > 0), whichever kernels run, against the float64 oracle."""
import numpy as np
import pytest

from gpu_common import TOL, gpu_outputs, gpu_scan, gpu_scan_gated, normwise, oracle_outputs
from paper_2406_12580_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

# team kernels: one tile, whole chains a team with several tiles, the look-back (near,
# far, with a ragged last tile); serial kernels, narrow ones among them in bfloat16
SHAPES = [(3, 100, 72), (310, 300, 24), (3, 1500, 136), (1, 6000, 8), (520, 60, 40), (800, 60, 40)]


def put(inp, name, at, v):
    getattr(inp, name)[at] = v
    if inp.cfg.io == I.BF16:  # v: not finite, or 1
        inp.bits[name][at] = np.float32(v).view(np.uint32) >> 16


def same(got, want, tol, name):
    finite = np.isfinite(want)
    assert np.array_equal(np.isnan(got), np.isnan(want)), name
    assert np.array_equal(got[~finite & ~np.isnan(want)], want[~finite & ~np.isnan(want)]), name
    assert normwise(got[finite], want[finite]) <= tol, name


@pytest.mark.parametrize("io", [I.F32, I.BF16])
@pytest.mark.parametrize("gated", [False, True])
@pytest.mark.parametrize("B,L,D", SHAPES)
def test_infinite_states(B, L, D, gated, io):
    """An infinite x, h0, or both signs of them in different rows and channels."""
    cfg = I.ScanConfig("infinite states", io=io, seed=51, gated=gated, B=B, L=L, D=D, random_h0=True)
    inp = I.make_scan_inputs(cfg)
    for n, (t, v) in enumerate(((0, np.inf), (7, -np.inf), (L // 3, np.inf), (L - 1, -np.inf))):
        put(inp, "x", (n % B, t, n), v)
        put(inp, "gl", (n % B, t, D + n), 1.0)  # bfloat16's i x is formed as (x/2) tanh(iota/2) + x/2
    inp.h0[0, 5], inp.h0[B - 1, 6] = np.inf, -np.inf
    got = gpu_outputs(gpu_scan_gated(inp, with_bwd=False) if gated else gpu_scan(inp, with_bwd=False))
    want = oracle_outputs(inp)
    assert not np.isfinite(want["h"]).all()
    for k in ("h", "h_last"):
        same(got[k], want[k], TOL[io], k)


@pytest.mark.parametrize("io", [I.F32, I.BF16])
@pytest.mark.parametrize("gated", [False, True])
@pytest.mark.parametrize("B,L,D", SHAPES)
def test_infinite_adjoints(B, L, D, gated, io):
    """An infinite dh (dy) or dh_last reaches every step before it."""
    cfg = I.ScanConfig("infinite adjoints", io=io, seed=52, gated=gated, B=B, L=L, D=D,
                       random_h0=True, random_dh_last=True)
    inp = I.make_scan_inputs(cfg)
    for n, (t, v) in enumerate(((0, np.inf), (L // 2, -np.inf), (2 * L // 3, np.inf), (L - 1, np.inf))):
        put(inp, "dh", (n % B, t, n), v)
    inp.dh_last[0, 5], inp.dh_last[B - 1, 6] = np.inf, -np.inf
    got = gpu_outputs(gpu_scan_gated(inp) if gated else gpu_scan(inp))
    want = oracle_outputs(inp)
    assert not np.isfinite(want["dx"]).all()
    for k in ("h", "dx", "dh0") + (("dz",) if gated else ()):
        same(got[k], want[k], TOL[io], k)
    # the gates' gradients: infinite in the same places (a sign is that of a difference)
    assert np.array_equal(np.isfinite(got["dgl"]), np.isfinite(want["dgl"]))
    assert np.array_equal(np.isfinite(got["dlam"]), np.isfinite(want["dlam"]))


@pytest.mark.parametrize("io", [I.F32, I.BF16])
@pytest.mark.parametrize("gated", [False, True])
@pytest.mark.parametrize("B,L,D", SHAPES)
def test_nans_stay_in_their_channels(B, L, D, gated, io):
    """A NaN in x, a logit or dh reaches what depends on it and nothing else."""
    cfg = I.ScanConfig("nan", io=io, seed=53, gated=gated, B=B, L=L, D=D, random_h0=True)
    inp = I.make_scan_inputs(cfg)
    put(inp, "x", (0, L // 2, 0), np.nan)
    put(inp, "gl", (B - 1, L // 3, 1), np.nan)
    put(inp, "dh", (B // 2, 2 * L // 3, 2), np.nan)
    got = gpu_outputs(gpu_scan_gated(inp) if gated else gpu_scan(inp))
    want = oracle_outputs(inp)
    for k in ("h", "h_last", "dx", "dgl", "dlam", "dh0") + (("dz",) if gated else ()):
        assert np.isnan(want[k]).any() or k == "dh0"
        same(got[k], want[k], TOL[io], k)


@pytest.mark.parametrize("io", [0, 1])
@pytest.mark.parametrize("K", [1, 3, 9])
def test_infinite_steps(K, io):
    """blr_steps and blr_step on infinite inputs and states, gates open and nearly closed."""
    from paper_2406_12580_gb300 import blr_step, blr_steps
    B, D = 5, 24
    g = torch.Generator(device="cuda").manual_seed(K)
    rand = lambda *s: torch.randn(*s, device="cuda", generator=g)  # noqa: E731
    dtype = (torch.float32, torch.bfloat16)[io]
    h, x, gl, lam = rand(B, D), rand(B, K, D), rand(B, K, 2 * D), rand(D) - 3.0
    x[0, 0, 0], x[1, K - 1, 1], x[2, 0, 2], h[3, 3], h[4, 4] = np.inf, -np.inf, np.inf, np.inf, -np.inf
    gl[0, 0, D], gl[1, K - 1, D + 1], gl[2, 0, D + 2] = -2.0, -1.0, 3.0
    x, gl = x.to(dtype), gl.to(dtype)
    ref, want = h.double(), []
    r, i = torch.sigmoid(gl.double()).chunk(2, dim=-1)
    log_a = -torch.nn.functional.softplus(lam.double()) * r
    for k in range(K):
        ref = torch.exp(log_a[:, k]) * ref + torch.sqrt(-torch.expm1(2 * log_a[:, k])) * i[:, k] * x[:, k].double()
        want.append(ref)
    out, seq = torch.empty_like(h), torch.empty_like(x)
    blr_steps(B, K, D, io, 0, 1.0, h, x, gl, lam, out, seq)
    tol = TOL[I.BF16 if io else I.F32]
    same(out.double().cpu().numpy(), ref.cpu().numpy(), tol, "h")
    same(seq.double().cpu().numpy(), torch.stack(want, 1).cpu().numpy(), tol, "h_seq")
    if K == 1:
        blr_step(B, D, io, 1.0, h, x[:, 0].contiguous(), gl[:, 0].contiguous(), lam, out)
        same(out.double().cpu().numpy(), ref.cpu().numpy(), tol, "step")
