"""Weights-only convolution at the edges of its forms: the tiles of 64 filters beyond the first wave (two CTAs on an SM, one
operand stage of 128 elements) at row lengths of one and several stages and one more or less, more filters than a tile at short
rows, and windows of so many elements that a stage lies in one channel."""
import pytest

import dab_synth
from test_gpu_wbin import _check, dab  # noqa: F401  (the fixture and the bound against the checker)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,C,H,W,Cout,k,stride,pad", [
    (5, 1, 64, 63, 5, 1, 1, 0),       # rows of one value
    (9, 3, 46, 47, 64, 3, 1, 1),      # 27 values, a mask word; 152 tiles
    (9, 96, 46, 46, 3, 1, 1, 0),      # 96 values
    (5, 2, 64, 64, 130, 4, 1, 0),     # 32 values, three tiles of filters
    (20, 16, 32, 31, 63, 3, 1, 1),    # 144 values: a full stage and one of 16
    (20, 14, 32, 32, 33, 3, 1, 1),    # 126 values
    (3, 1, 90, 90, 20, 16, 1, 0),     # 256 values of one channel
    (2, 1, 60, 130, 9, 31, 1, 0),     # 961 values: windows of more than a stage, within the first wave
    (1, 2, 80, 81, 9, 50, 3, 0)])     # 5000 values
def test_forms(dab, N, C, H, W, Cout, k, stride, pad):  # noqa: F811
    x = dab_synth.relu_activations((N, C, H, W), 0.5, stream=640 + C + k)
    w = dab_synth.normal((Cout, C * k * k), 0.05, stream=650 + C + k)
    _check(dab, x, w, k, k, (stride, stride), (pad, pad))
