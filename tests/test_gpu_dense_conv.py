"""The tiled full-precision convolution against the CPU checker, equal to the bit, at the edges of its tiles: position
and filter remainders of the three tile shapes, rows shorter than, equal to and just beyond a chunk of taps, padding,
and windows that cover the whole (padded) image, which are staged along the taps."""
import numpy as np
import pytest
import torch

import oracle
from parity_util import to_dev

pytestmark = pytest.mark.gpu

CASES = [  # N, C, H, W, Cout, kh, kw, stride, pad
    (3, 1, 80, 81, 64, 4, 4, 1, 0),      # 128 x 64 tiles, 16 taps (one chunk)
    (5, 2, 64, 63, 66, 3, 3, 1, 1),      # ... two tiles of filters, the second of 2; 18 taps; padding
    (7, 3, 61, 60, 96, 5, 3, 1, 2),      # 128 x 48 tiles, 45 taps
    (9, 5, 93, 95, 33, 3, 3, 2, 1),      # 128 x 48, one ragged tile of filters, stride 2
    (1, 1, 9, 9, 1, 2, 2, 1, 0),         # small: one position tile, one filter
    (2, 13, 11, 7, 17, 3, 5, 2, 1),      # small: 195 taps, ragged both ways
    (1, 64, 5, 5, 18, 1, 1, 1, 0),       # small: exactly one chunk of 64 taps
    (33, 65, 1, 1, 19, 1, 1, 1, 0),      # fully connected, 65 taps, 33 images
    (31, 6, 4, 5, 15, 6, 7, 1, 1),       # window over the padded image
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_dense_convolution_tiles(case):
    import paper_1804_02941_b200 as dab
    N, C, H, W, Cout, kh, kw, stride, pad = case
    rng = np.random.default_rng(sum(case))
    x = rng.standard_normal((N, C, H, W)).astype(np.float32)
    x[rng.random(x.shape) < 0.3] = 0.0
    layer = {"kind": "conv_dense", "w": rng.standard_normal((Cout, C * kh * kw)).astype(np.float32), "kh": kh, "kw": kw,
             "stride": (stride, stride), "pad": (pad, pad), "bias": rng.standard_normal(Cout).astype(np.float32)}
    y = dab.dab_network_forward(dab.Network([layer]), to_dev(x))
    torch.cuda.synchronize()
    want, _ = oracle.network_layer(layer, x, None)
    assert np.array_equal(y.cpu().numpy(), want)
