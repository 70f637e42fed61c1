"""The tensor-core contraction of long rows, tiles of 128 x 128: row and column remainders, row lengths around its stages of 256 bits, both output layouts.  Rows at the edges of tiles against the CPU checker (counts bit
for bit, outputs within 1e-5 relative: one rounding of the same fp64 sum each), everything bit for bit against population counts."""
import numpy as np
import pytest
import torch

import dab_synth
import oracle
from parity_util import rel_close, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,n", [(1793, 2690, 2048), (1900, 2433, 2303), (2000, 2570, 2304), (1665, 2817, 4097), (2049, 2313, 2177),
                                   (5000, 1030, 16384)])
def test_long_rows(M, N, n):
    import paper_1804_02941_b200 as dab
    oracle.set_threads(16)
    A = dab_synth.relu_activations((M, n), 0.6, stream=700 + M)
    B = dab_synth.normal((N, n), 0.05, stream=800 + N)
    a, b = dab.dab_binarize(to_dev(A)), dab.dab_binarize(to_dev(B))
    out = {}
    for path in (dab.CONTRACT_POPC, dab.CONTRACT_AUTO):
        dab.dab_set_contraction(path)
        try:
            out[path] = (*dab.dab_binary_gemm(a, b, want_p11=True), dab.dab_binary_conv(to_dev(A).view(M, n, 1, 1), b, 1, 1).view(M, N))
        finally:
            dab.dab_set_contraction(dab.CONTRACT_AUTO)
    torch.cuda.synchronize()
    assert dab.dab_contraction_wait_failures() == 0
    for popc, tensor in zip(*out.values()):
        assert torch.equal(popc, tensor)
    C, p11, conv = out[dab.CONTRACT_AUTO]
    assert torch.equal(C, conv)
    rows = sorted({0, 1, 127, 128, 129, 255, 256, 257, M - 1, M - 130, M // 256 * 256 - 1, M // 256 * 256})
    ra, rb = oracle.binarize(A[rows]), oracle.binarize(B)
    ref, refP = oracle.gemm(ra.e, ra.alpha, ra.beta, rb.e, rb.alpha, rb.beta)
    assert np.array_equal(p11[rows].cpu().numpy(), refP)
    assert rel_close(C[rows].cpu().numpy(), ref).all()
