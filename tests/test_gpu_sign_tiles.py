"""The sign coder of patches at the edges of its tiles, against the CPU checker: 32 channels fill whole words, so channel
counts around multiples of 32; windows of every shape it unrolls or loops over; tiles of one row, of one column and wider
than a ballot; strides, paddings, negative zeros and non-finite values."""
import numpy as np
import pytest
import torch

import oracle
from parity_util import check_coded, to_dev

pytestmark = pytest.mark.gpu

CASES = [  # N, C, H, W, kh, kw, stride, pad
    (2, 31, 9, 9, 3, 3, 1, 1),
    (1, 32, 33, 30, 3, 3, 1, 1),     # 30 output columns: exactly one ballot
    (2, 33, 5, 57, 3, 3, 1, 1),      # two tiles across, the second ragged
    (3, 65, 7, 7, 3, 3, 2, 1),
    (1, 3, 40, 40, 5, 5, 1, 2),
    (2, 37, 8, 11, 1, 1, 1, 0),      # one bit per channel
    (2, 40, 13, 10, 1, 1, 2, 0),
    (1, 20, 7, 7, 7, 7, 1, 0),       # one patch per image
    (1, 5, 6, 70, 2, 32, 1, 0),      # a window as wide as a ballot
    (1, 4, 5, 60, 2, 33, 3, 1),      # and one wider
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_sign_patches(case):
    import paper_1804_02941_b200 as dab
    N, C, H, W, kh, kw, stride, pad = case
    rng = np.random.default_rng(sum(case))
    x = rng.standard_normal((N, C, H, W)).astype(np.float32)
    x[rng.random(x.shape) < 0.2] = 0.0
    x[rng.random(x.shape) < 0.05] = -0.0
    x[0, C - 1, H - 1, W - 1] = np.nan
    x[0, 0, 0, 0] = np.inf
    desc = dab.make_desc(x.shape, 4, kh, kw, (stride, stride), (pad, pad))
    ho, wo = dab.dab_conv_output_size(desc)
    P, n = N * ho * wo, C * kh * kw
    new = lambda *s, dtype=torch.int32: torch.full(s, -7, dtype=dtype, device="cuda")
    c = dab.Coded(new(P, dab.dab_default_ld(n) + 4), new(P), new(P, dtype=torch.float32), new(P, dtype=torch.float32), new(P), n)
    dab.dab_sign_patches(desc, to_dev(x), c.K, c.alpha, c.beta, c.mask, c.flags)
    torch.cuda.synchronize()
    check_coded(c, oracle.sign_code(oracle.im2col(x, kh, kw, (stride, stride), (pad, pad))), n)
