"""GPU: scans whose forward and backward run in different forms, against the oracle:
float32 ones whose forward runs on the team kernels and whose backward on the serial
ones, on both sides of the lines between (tiles in the local order and with the
look-back, whole and ragged last ones), and gated bfloat16 ones at the narrow form's."""
import pytest

from gpu_common import TOL, compare, gpu_outputs, gpu_scan, gpu_scan_gated, normwise, oracle_outputs
from paper_2406_12580_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("gated", [False, True])
@pytest.mark.parametrize("B,L,D", [(455, 800, 32), (456, 799, 32), (456, 800, 32), (228, 801, 64),
                                   (122, 1024, 128), (416, 800, 32), (488, 385, 32), (244, 400, 64),
                                   (244, 384, 64), (460, 810, 24), (58, 800, 256)])
def test_team_forward_serial_backward(B, L, D, gated):
    cfg = I.ScanConfig("mixed", io=I.F32, seed=B + L, gated=gated, B=B, L=L, D=D, random_h0=True,
                       random_dh_last=True)
    inp = I.make_scan_inputs(cfg)
    buf, want = (gpu_scan_gated if gated else gpu_scan)(inp), oracle_outputs(inp)
    compare(inp, gpu_outputs(buf), want)
    (buf.bwd_gated if gated else buf.bwd)()  # again on the same workspace
    torch.cuda.synchronize()
    for k, v in gpu_outputs(buf).items():
        assert normwise(v, want[k]) <= TOL[I.F32], k


@pytest.mark.parametrize("B,L", [(1976, 23), (1977, 23), (1977, 100), (1977, 101)])
def test_bf16_merge_by_chains(B, L):
    """bfloat16 with the merge at the line between the wide and the narrow forward."""
    cfg = I.ScanConfig("merge", io=I.BF16, seed=B + L, gated=True, B=B, L=L, D=64, random_h0=True)
    inp = I.make_scan_inputs(cfg)
    compare(inp, gpu_outputs(gpu_scan_gated(inp)), oracle_outputs(inp))
