"""The population-count contraction where a cluster splits the row length, against the CPU checker: 2, 4 and 8 members, shares
that end inside the last member and members left without words; one to 17 activation rows (the two tile heights); both
output layouts.  Counts bit for bit, outputs within 1e-5 relative (one rounding of the same fp64 sum each)."""
import numpy as np
import pytest
import torch

import dab_synth
import oracle
from parity_util import rel_close, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,n", [(1, 512, 12544), (16, 70, 800), (17, 64, 770), (225, 256, 1600), (100, 1500, 4608),
                                   (33, 3000, 16384), (900, 513, 380), (64, 130, 752), (2, 1, 16383)])
def test_split_gemm(M, N, n):
    import paper_1804_02941_b200 as dab
    oracle.set_threads(16)
    A = dab_synth.relu_activations((M, n), 0.6, stream=500 + M)
    B = dab_synth.normal((N, n), 0.05, stream=600 + N)
    ra, rb = oracle.binarize(A), oracle.binarize(B)
    ref, refP = oracle.gemm(ra.e, ra.alpha, ra.beta, rb.e, rb.alpha, rb.beta)
    a, b = dab.dab_binarize(to_dev(A)), dab.dab_binarize(to_dev(B))
    dab.dab_set_contraction(dab.CONTRACT_POPC)
    try:
        got, p11 = dab.dab_binary_gemm(a, b, want_p11=True)
        conv = dab.dab_binary_conv(to_dev(A).view(M, n, 1, 1), b, 1, 1)   # the NCHW layout: one position per image
    finally:
        dab.dab_set_contraction(dab.CONTRACT_AUTO)
    torch.cuda.synchronize()
    assert np.array_equal(p11.cpu().numpy(), refP)
    assert rel_close(got.cpu().numpy(), ref).all()
    assert torch.equal(conv.view(M, N), got)
