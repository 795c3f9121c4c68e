"""GPU: the team kernels and the narrow serial ones at the edges of their tiles,
against the oracle.

Tiles are up to 128 steps, slices 16 steps a warp; a chain is 32 float32 or 64
bfloat16 channels of one batch row. The bounds are those of the other parity
tests (``gpu_common``): the kernels hold states, carries and products in
float32 and round each output once.
"""
import numpy as np
import pytest

from gpu_common import (TOL, compare, gpu_outputs, gpu_scan, gpu_scan_gated, normwise,
                        oracle_outputs)
from paper_2406_12580_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

EDGES = [
    # one slice, a slice and a step, a full tile, a full tile and a step
    dict(B=2, L=16, D=8, random_h0=True, random_dh_last=True),
    dict(B=3, L=17, D=72),
    dict(B=2, L=128, D=64, random_dh_last=True),
    dict(B=2, L=129, D=136, random_h0=True),
    # several tiles a chain: a ragged last one, and a look-back several tiles deep
    dict(B=2, L=1000, D=200, random_h0=True, random_dh_last=True, decay=(0.99, 0.9999)),
    dict(B=1, L=6000, D=8, random_h0=True, random_dh_last=True),
    # more chains than teams in the local order, and with the look-back
    dict(B=310, L=150, D=24, random_h0=True),
    dict(B=401, L=700, D=8, random_dh_last=True),
    # teams that change their channel group from tile to tile
    dict(B=2, L=300, D=1400, random_h0=True, random_dh_last=True),
    # the general e^l - 1 branch
    dict(B=4, L=200, D=40, decay=(0.05, 0.95), c=3.0, random_h0=True, random_dh_last=True),
    # bfloat16: the serial kernels' narrow form, by few chains (a step, a kept
    # state's and a box's steps and one more, several boxes; a channel tail, an odd
    # number of groups) and by few channels; and the general branch in it
    dict(B=304, L=1, D=64, random_h0=True, random_dh_last=True),
    dict(B=305, L=8, D=8, random_dh_last=True),
    dict(B=304, L=9, D=40, random_h0=True),
    dict(B=170, L=16, D=120, random_h0=True, random_dh_last=True),
    dict(B=110, L=17, D=160),
    dict(B=330, L=100, D=72, random_h0=True, random_dh_last=True, decay=(0.99, 0.9999)),
    dict(B=2100, L=33, D=24, random_h0=True, random_dh_last=True),
    dict(B=320, L=50, D=56, decay=(0.05, 0.95), c=3.0, random_h0=True, random_dh_last=True),
    # only the backward narrow, and with the merge only the forward
    dict(B=1000, L=41, D=64, random_h0=True, random_dh_last=True),
    dict(B=1830, L=23, D=64, random_h0=True),
    dict(B=620, L=170, D=160, random_dh_last=True),
]


@pytest.mark.parametrize("io", [I.F32, I.BF16])
@pytest.mark.parametrize("mode", ["plain", "gated", "varlen"])
@pytest.mark.parametrize("case", range(len(EDGES)))
def test_team_edges(case, mode, io):
    cfg = I.ScanConfig(f"team {case} {mode}", io=io, seed=1300 + case, gated=mode == "gated",
                       **EDGES[case])
    inp = I.make_scan_inputs(cfg)
    if mode == "plain":
        compare(inp, gpu_outputs(gpu_scan(inp)), oracle_outputs(inp))
        return
    if mode == "gated":
        compare(inp, gpu_outputs(gpu_scan_gated(inp)), oracle_outputs(inp))
        return
    import oracle
    from paper_2406_12580_gb300.device import ScanBuffers
    lengths = np.random.default_rng(case).integers(0, cfg.L + 1, size=cfg.B).astype(np.int32)
    lengths[0] = cfg.L
    lengths[-1] = min(16, cfg.L)
    buf = ScanBuffers.from_inputs(inp)
    for t in (buf.h, buf.dx, buf.dgl):
        t.fill_(7.0)  # the padding is not written
    lt = torch.from_numpy(lengths).cuda()
    buf.fwd_varlen(lt)
    buf.bwd_varlen(lt)
    torch.cuda.synchronize()
    orc = oracle.load()
    h, h_last = orc.fwd_varlen(lengths, inp.x, inp.gl, inp.lam, inp.h0, c=cfg.c)
    dx, dgl, dlam, dh0 = orc.bwd_varlen(lengths, inp.dh, inp.x, inp.gl, inp.lam, inp.h0,
                                        inp.dh_last, c=cfg.c)
    got = gpu_outputs(buf)
    real = (np.arange(cfg.L)[None] >= cfg.L - lengths[:, None])[..., None]
    for k, want in (("h", h), ("dx", dx), ("dgl", dgl)):
        mask = np.broadcast_to(real, want.shape)
        assert (got[k][~mask] == 7.0).all(), k
        assert normwise(got[k][mask], want[mask]) <= TOL[io], k
    for k, want in (("h_last", h_last), ("dlam", dlam), ("dh0", dh0)):
        assert normwise(got[k], want) <= TOL[io], k


@pytest.mark.parametrize("io", [I.F32, I.BF16])
@pytest.mark.parametrize("mode", ["plain", "gated", "varlen"])
def test_backward_again_on_one_workspace(mode, io):
    """Backwards that follow one forward find their look-back records empty,
    whatever the workspace held before (zeros would read as published states)."""
    cfg = I.ScanConfig(f"again {mode}", io=io, seed=77, gated=mode == "gated", B=3, L=1500, D=136,
                       random_h0=True, random_dh_last=True)
    inp = I.make_scan_inputs(cfg)
    from paper_2406_12580_gb300.device import ScanBuffers
    buf = ScanBuffers.from_inputs(inp)
    lengths = torch.tensor([cfg.L, 1025, 300], dtype=torch.int32, device="cuda")
    first, want = None, None if mode == "varlen" else oracle_outputs(inp)
    for fill in (0, 255, 0):
        buf.ws.fill_(fill)
        if mode == "varlen":
            buf.h.zero_(), buf.dx.zero_(), buf.dgl.zero_()
            buf.fwd_varlen(lengths)
        else:
            (buf.fwd_gated if mode == "gated" else buf.fwd)()
        for _ in range(4):
            if mode == "varlen":
                buf.bwd_varlen(lengths)
            else:
                (buf.bwd_gated if mode == "gated" else buf.bwd)()
            torch.cuda.synchronize()
            got = gpu_outputs(buf)
            if mode != "varlen":
                for k, v in want.items():
                    assert normwise(got[k], v) <= TOL[io], k
            first = first or got
            for k, v in got.items():
                assert v is None or normwise(v, first[k]) <= TOL[io], k

def test_scratch_call_takes_the_local_order():
    """A problem whose look-back records do not fit the library's scratch still
    runs there: the forward without a workspace takes the local order."""
    from paper_2406_12580_gb300 import (BLR_OK, Desc, blr_scan_fwd_noalloc, blr_workspace_bytes,
                                        blr_workspace_status)
    B, L, D = 400, 33000, 32   # 400 float32 chains
    desc = Desc(B, L, D, 0, 1.0)
    assert blr_workspace_bytes(desc) > 128 << 20
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn(B, L, D, device="cuda", generator=g)
    gl = torch.randn(B, L, 2 * D, device="cuda", generator=g)
    lam = torch.from_numpy(I.lambda_from_decay(np.linspace(0.9, 0.999, D)).astype(np.float32)).cuda()
    h, h2 = torch.empty_like(x), torch.empty_like(x)
    h_last, h_last2 = (torch.empty(B, D, device="cuda") for _ in range(2))
    from paper_2406_12580_gb300 import blr_scan_fwd
    ws = torch.empty(blr_workspace_bytes(desc), dtype=torch.uint8, device="cuda")
    blr_scan_fwd(desc, x, gl, lam, None, h, h_last, ws)
    blr_scan_fwd_noalloc(desc, x, gl, lam, None, h2, h_last2)
    assert blr_workspace_status(desc, None) == BLR_OK
    # the two orders differ in the order of float32 compositions only
    assert normwise(h2.cpu().numpy(), h.cpu().numpy()) <= TOL[I.F32]
    assert normwise(h_last2.cpu().numpy(), h_last.cpu().numpy()) <= TOL[I.F32]


@pytest.mark.parametrize("B,L,D", [(1, 20, 8), (12, 300, 72), (127, 150, 128), (250, 40, 16)])
def test_small_gated_bf16_gradients_are_the_separate_merges(B, L, D):
    """d Lambda and dh0 of small bfloat16 problems with the merge are those of
    the plain scan given dh = dy SiLU(z) rounded to bfloat16. Both sides round the
    same float32 product but for its last bits (2e-6 of 2^-9: one value in a
    thousand lands on the other side, 2^-9 sqrt(1e-3) = 6e-5 of the sums; without
    the rounding, or with tanh for the sigmoid, they differ by 1e-3 and more)."""
    from paper_2406_12580_gb300 import (BLR_BF16, Desc, blr_scan_bwd, blr_scan_bwd_gated,
                                        blr_scan_fwd, blr_scan_fwd_gated, blr_workspace_bytes)
    g = torch.Generator(device="cuda").manual_seed(B + L + D)
    rand = lambda *s: torch.randn(*s, device="cuda", generator=g).bfloat16()  # noqa: E731
    x, z, dy, gl = rand(B, L, D), rand(B, L, D), rand(B, L, D), rand(B, L, 2 * D)
    h0 = torch.randn(B, D, device="cuda", generator=g)
    lam = torch.from_numpy(I.lambda_from_decay(np.linspace(0.9, 0.999, D)).astype(np.float32)).cuda()
    desc = Desc(B, L, D, BLR_BF16, 1.0)
    ws = torch.empty(blr_workspace_bytes(desc), dtype=torch.uint8, device="cuda")
    y, dx, dz, dgl = (torch.empty_like(t) for t in (x, x, z, gl))
    got, want = ([torch.empty_like(lam), torch.empty_like(h0)] for _ in range(2))
    blr_scan_fwd_gated(desc, x, gl, lam, h0, z, y, None, ws)
    blr_scan_bwd_gated(desc, dy, None, x, gl, lam, h0, z, dx, dgl, dz, *got, ws)
    dh = (dy.float() * torch.nn.functional.silu(z.float())).bfloat16()
    blr_scan_fwd(desc, x, gl, lam, h0, y, None, ws)
    blr_scan_bwd(desc, dh, None, x, gl, lam, h0, dx, dgl, *want, ws)
    for a, b in zip(got, want):
        assert (a - b).norm().item() <= 2e-4 * b.norm().item()
