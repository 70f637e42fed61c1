"""Max pooling against the CPU checker, equal to the bit: windows that the kernels unroll and others, strides, paddings (also windows in the
padding alone), NaN, and zeros of both signs."""
import numpy as np
import pytest
import torch

import oracle
from parity_util import to_dev

pytestmark = pytest.mark.gpu

POOL = [(3, 5, 17, 19, 3, 2, 0), (2, 7, 14, 15, 3, 1, 1), (2, 3, 12, 12, 2, 2, 0), (4, 9, 7, 7, 7, 7, 0), (2, 3, 9, 11, 5, 3, 2), (1, 1, 3, 3, 3, 1, 2),
        (2, 3, 5, 6, 2, 1, 3), (2, 2, 6, 5, 3, 2, 4), (2, 3, 9, 8, 6, 1, 7), (2, 3, 4, 5, 1, 1, 2),   # windows in the padding alone
        (1, 1, 1500, 3000, 2, 1, 0),   # an output's row by a 64-bit division
        (2, 3, 60000, 2, 2, 2, 0)]     # its plane as well


@pytest.mark.parametrize("case", POOL, ids=lambda c: "x".join(map(str, c)))
def test_pooling(case):
    import paper_1804_02941_b200 as dab
    N, C, H, W, k, stride, pad = case
    rng = np.random.default_rng(sum(case))
    x = np.where(rng.random((N, C, H, W)) < 0.3, rng.choice([0.0, -0.0], (N, C, H, W)), rng.standard_normal((N, C, H, W))).astype(np.float32)
    x[0, 0, 1, 1] = np.nan
    layer = {"kind": "maxpool", "kh": k, "kw": k, "stride": (stride, stride), "pad": (pad, pad)}
    y = dab.dab_network_forward(dab.Network([layer]), to_dev(x))
    torch.cuda.synchronize()
    want, _ = oracle.network_layer(layer, x, None)
    assert np.array_equal(y.cpu().numpy().view(np.uint32), np.asarray(want, np.float32).view(np.uint32))


@pytest.mark.parametrize("N,C,k", [(3, 5, 3), (2, 7, 2), (2, 3, 5), (1, 70000, 2)])   # the last: a plane's channel by a 64-bit division
def test_layers_behind_pooling(N, C, k):
    # another scale and shift in every channel, small multiples of powers of two: nothing is rounded
    import paper_1804_02941_b200 as dab
    rng = np.random.default_rng(N + C + k)
    x = rng.integers(-64, 65, (N, C, k + 1, k + 2)).astype(np.float32)
    layers = [{"kind": "maxpool", "kh": k, "kw": k, "stride": (1, 1), "pad": (0, 0)}, {"kind": "affine", "scale": (1.0 + np.arange(C) % 97).astype(np.float32),
              "shift": (0.25 * rng.integers(-100, 100, C)).astype(np.float32)}, {"kind": "relu"}]
    y = dab.dab_network_forward(dab.Network(layers), to_dev(x))
    torch.cuda.synchronize()
    assert np.array_equal(y.cpu().numpy(), oracle.network_forward(layers, x))
