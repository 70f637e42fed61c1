"""Full-precision convolutions of few filters: tiles of 8 and 16 filters and the thread per output, at the filter and tap counts they
change at, with padding, strides, a bias and the elementwise layers behind.  Bit for bit against the CPU checker."""
import numpy as np
import pytest
import torch

import dab_synth
import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Cout", [1, 2, 3, 8, 9, 16, 17])
@pytest.mark.parametrize("C,H,W,k,stride,pad", [(2, 71, 70, 4, 1, 0), (3, 70, 73, 3, 1, 1), (11, 69, 71, 3, 1, 2), (1, 140, 139, 5, 2, 2)])
def test_few_filters(C, H, W, k, stride, pad, Cout):
    import paper_1804_02941_b200 as dab
    oracle.set_threads(16)
    N = 5
    x = dab_synth.normal((N, C, H, W), 1.0, stream=C + k)
    w = dab_synth.normal((Cout, C * k * k), 0.3, stream=C + k + 1)
    bias = dab_synth.normal((Cout,), 0.5, stream=C + k + 2)
    scale, shift = dab_synth.normal((Cout,), 1.0, stream=5), dab_synth.normal((Cout,), 1.0, stream=6)
    conv = {"kind": "conv_dense", "w": w, "bias": bias, "kh": k, "kw": k, "stride": (stride, stride), "pad": (pad, pad), "Cout": Cout}
    net = dab.Network([conv, {"kind": "affine", "scale": scale, "shift": shift}, {"kind": "relu"}])
    got = dab.dab_network_forward(net, torch.from_numpy(x).cuda()).cpu().numpy()
    ref = oracle.relu(oracle.affine(oracle.conv_dense(x, w, k, k, (stride, stride), (pad, pad), bias), scale, shift))
    assert got.shape == ref.shape and np.array_equal(got, ref)
