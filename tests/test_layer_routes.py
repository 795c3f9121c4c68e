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
