"""CPU: which calls of the gated layer may take the library's kernels."""
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
