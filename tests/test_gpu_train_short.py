"""The training step of short filters, which get a warp each: forward at the ends of the lengths of either coder and at few and many
filters, backward on both sides of where a filter gets a warp instead of a CTA.  Against the CPU checker; in place as well."""
import numpy as np
import pytest
import torch

import dab_synth
import oracle
from parity_util import rel_close, to_dev, unpack, words

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,n", [(3, 2), (70, 31), (9, 32), (4000, 33), (5, 255), (300, 256), (288, 256), (3000, 257), (3000, 512),
                                    (324, 289), (326, 290), (20, 513)])
def test_step_matches_checker(rows, n):
    import paper_1804_02941_b200 as dab
    oracle.set_threads(16)
    W = dab_synth.normal((rows, n), 0.5, stream=960 + n, mean=0.04)
    W[0] = 0.3                                          # constant
    W[1] = np.sign(W[1]) * 0.25                         # two values
    g = dab_synth.normal((rows, n), 1.0, stream=970 + n)
    Wc_r, e_r, K_r, a_r, b_r, f_r, Wt_r = oracle.train_forward(W)
    _, gw_r = oracle.theorem4(Wc_r, e_r, K_r, grad_Wt=g)
    Wc, coded, Wt = dab.dab_binarize_train(to_dev(W))
    gw = dab.dab_binarize_backward(Wc, coded, to_dev(g))
    torch.cuda.synchronize()
    assert np.array_equal(Wc.cpu().numpy(), Wc_r)
    assert np.array_equal(coded.K.cpu().numpy(), K_r)
    assert np.array_equal(coded.flags.cpu().numpy().view(np.uint32), f_r)
    assert np.array_equal(unpack(words(coded.mask), n), e_r)
    assert rel_close(coded.alpha.cpu().numpy(), a_r).all() and rel_close(coded.beta.cpu().numpy(), b_r).all()
    assert rel_close(Wt.cpu().numpy(), Wt_r).all()
    assert rel_close(gw.cpu().numpy(), gw_r).all()


def test_in_place_without_dense_filters_or_flags():
    import ctypes as C
    import paper_1804_02941_b200 as dab
    rows, n, ld = 50, 100, 8                            # a mask row of 4 words in a stride of 8
    W = to_dev(dab_synth.normal((rows, n), 0.2, stream=990))
    Wc, coded, _ = dab.dab_binarize_train(W)
    m = torch.full((rows, ld), -1, dtype=torch.int32, device="cuda")
    K = torch.empty(rows, dtype=torch.int32, device="cuda")
    a, b = torch.empty(rows, device="cuda"), torch.empty(rows, device="cuda")
    p = lambda t: C.c_void_p(t.data_ptr())
    assert dab.lib().dab_binarize_train(p(W), rows, n, n, p(W), n, None, 0, p(K), p(a), p(b), p(m), ld, None, None) == 0
    torch.cuda.synchronize()
    assert torch.equal(W, Wc) and torch.equal(K, coded.K) and torch.equal(a, coded.alpha) and torch.equal(b, coded.beta)
    assert torch.equal(m[:, :4], coded.mask) and not m[:, 4:].any()
