"""Weights-only convolution whose stride steps over rows of the input: between the windows of neighbouring output rows nothing
is staged, and layers with wide windows fit shared memory for that reason only."""
import numpy as np
import pytest

import dab_synth
from test_gpu_wbin import _check, dab  # noqa: F401  (the fixture and the bound against the checker)

pytestmark = pytest.mark.gpu


# (N, C, H, W, Cout, kh, kw, stride, pad): the first three fit with one output row of one image in a tile; several images and
# rows per tile; windows lower than the stride by one and by many rows
@pytest.mark.parametrize("N,C,H,W,Cout,kh,kw,stride,pad", [
    (2, 4, 16, 247, 6, 16, 247, (32, 62), (8, 123)), (2, 5, 7, 298, 7, 7, 298, (30, 1), (3, 149)),
    (1, 11, 70, 288, 3, 5, 285, (29, 285), (0, 142)), (5, 6, 41, 9, 70, 3, 3, (4, 2), (0, 1)), (9, 40, 20, 20, 5, 1, 1, (7, 1), (0, 0))])
def test_strides_taller_than_the_window(dab, N, C, H, W, Cout, kh, kw, stride, pad):  # noqa: F811
    x = dab_synth.normal((N, C, H, W), 1.0, stream=610 + C).astype(np.float32)
    w = dab_synth.normal((Cout, C * kh * kw), 0.05, stream=620 + C)
    _check(dab, x, w, kh, kw, stride, pad)
