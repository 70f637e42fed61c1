"""Elementwise layers taken along by the layer before them, against the CPU checker, layer by layer on the tensors the GPU
produced (equal: an affine layer is rounded once here and twice there, which differs in about one value in 2^29; there are some 9 million,
of fixed seeds), and with and without kept layer outputs (bit for bit):
chains longer than one kernel takes, chains that begin a network or follow layers of the remembered tensor, several shortcuts
in one chain, planes that are not a multiple of four, and every kernel such a chain can hang on (dense convolution, both
contractions, pooling, the pass of its own)."""
import numpy as np
import pytest
import torch

import oracle
from parity_util import rel_close, to_dev

pytestmark = pytest.mark.gpu


def _chain(rng, c, cout):
    def conv(kind, co, ci, k, **more):
        return dict(kind=kind, w=(rng.standard_normal((co, ci * k * k)) * 0.1).astype(np.float32), kh=k, kw=k, stride=(1, 1),
                    pad=(k // 2, k // 2), Cout=co, **more)

    def affine(ch, **more):
        return dict(kind="affine", scale=rng.uniform(0.5, 1.5, ch).astype(np.float32),
                    shift=(rng.standard_normal(ch) * 0.1).astype(np.float32), **more)
    relu, save, add = dict(kind="relu"), dict(kind="save"), dict(kind="add")
    pool = dict(kind="maxpool", kh=3, kw=3, stride=(1, 1), pad=(1, 1))
    return [save, affine(c), relu, add, save,                                        # begins the network
            conv("conv_dense", cout, c, 3), relu, affine(cout), relu,
            conv("conv_dense", cout, c, 1, on_saved=True), affine(cout, on_saved=True), dict(relu, on_saved=True),
            add, relu, save, affine(cout),                                           # a pass of its own
            conv("conv_binary", cout, cout, 3), affine(cout), relu, affine(cout), add, save, affine(cout), add, relu,
            affine(cout), relu, affine(cout), affine(cout), add, save,               # longer than one kernel takes
            pool, affine(cout), save, relu,
            conv("conv_binary", 20, cout, 3), relu, save]


@pytest.mark.parametrize("N,C,H,W,Cout", [(1, 5, 7, 9, 33), (16, 3, 28, 28, 64), (2, 4, 11, 6, 300)])
def test_chains(N, C, H, W, Cout):
    import paper_1804_02941_b200 as dab
    oracle.set_threads(16)
    rng = np.random.default_rng(N + Cout)
    layers = _chain(rng, C, Cout)
    x = rng.standard_normal((N, C, H, W)).astype(np.float32)
    net = dab.Network(layers)
    shapes, c, saved_c = [], C, 0
    for l in layers:
        if l["kind"] == "save":
            saved_c = c
            shapes.append((c, H, W))
        elif l.get("on_saved"):
            saved_c = l.get("Cout", saved_c)
            shapes.append((saved_c, H, W))
        else:
            c = l.get("Cout", c)
            shapes.append((c, H, W))
    y, outs = dab.dab_network_forward(net, to_dev(x), keep_layers=True, layer_shapes=shapes)
    plain = dab.dab_network_forward(net, to_dev(x))
    torch.cuda.synchronize()
    assert torch.equal(y, plain)
    cur, saved = x, None
    for i, (l, got) in enumerate(zip(layers, outs)):
        got = got.cpu().numpy()
        want_cur, want_saved = oracle.network_layer(l, cur, saved)
        want = want_saved if l.get("on_saved") or l["kind"] == "save" else want_cur
        if l["kind"] == "conv_binary":
            assert rel_close(got, want).mean() > 0.999, i    # (a near-tie may go the other way)
        else:
            assert np.array_equal(got, want), (i, l["kind"])
        if l["kind"] == "save" or l.get("on_saved"):
            saved = got
        else:
            cur = got
    assert np.array_equal(plain.cpu().numpy(), cur)


@pytest.mark.parametrize("Cout", [20, 64, 300])
@pytest.mark.parametrize("contraction", ["CONTRACT_TENSOR", "CONTRACT_POPC"])
def test_a_tensor_stored_and_added_in_one_chain(contraction, Cout):
    # both contractions read what they have just written: the sum is twice the remembered tensor, then three times it
    import paper_1804_02941_b200 as dab
    rng = np.random.default_rng(Cout)
    conv = dict(kind="conv_binary", w=(rng.standard_normal((Cout, 27)) * 0.1).astype(np.float32), kh=3, kw=3, stride=(1, 1), pad=(1, 1), Cout=Cout)
    x = to_dev(rng.standard_normal((16, 3, 28, 28)).astype(np.float32))
    dab.dab_set_contraction(getattr(dab, contraction))
    try:
        once = dab.dab_network_forward(dab.Network([conv]), x)
        y = dab.dab_network_forward(dab.Network([conv, dict(kind="save"), dict(kind="add"), dict(kind="add")]), x)
    finally:
        dab.dab_set_contraction(dab.CONTRACT_AUTO)
    torch.cuda.synchronize()
    assert torch.equal(y, (once + once) + once)
