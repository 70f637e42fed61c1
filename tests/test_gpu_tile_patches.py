"""The tile coder of patches at the edges of its ranges, against the CPU checker: channel counts around a quadruple, a mask
word, its two table sizes and its two list types; windows up to 32 pixels; strides, paddings wider than the window, tiles
of one row, of one column and ragged ones; and inputs that leave a patch 1 to some thousand values to sort."""
import numpy as np
import pytest
import torch

import oracle
from parity_util import check_coded, to_dev

pytestmark = pytest.mark.gpu

CASES = [  # C, H, W, kh, kw, stride, pad
    (29, 9, 35, 3, 3, 1, 1),     # n = 261; two tiles across
    (33, 6, 5, 3, 3, 1, 1),
    (64, 18, 7, 3, 3, 2, 0),
    (170, 5, 6, 3, 3, 1, 1),     # n = 1530: the longest of the smaller tables
    (171, 5, 6, 3, 3, 1, 1),
    (256, 4, 5, 3, 3, 1, 1),     # channels in 8 bits
    (257, 4, 5, 3, 3, 1, 1),     # in 16
    (512, 4, 4, 3, 3, 2, 1),     # the mantissas of a pixel fill 32 bits
    (11, 8, 9, 5, 5, 1, 2),      # n = 275
    (130, 6, 5, 2, 2, 1, 1),
    (259, 1, 40, 1, 1, 1, 0),    # one pixel per patch, one row
    (255, 9, 3, 8, 4, 1, 4),     # 32 pixels, some windows in the padding alone, n = 8160
    (100, 20, 1, 3, 1, 1, 0),    # one column
]


def _images(rng, C, H, W):
    size = (C, H, W)
    x = [rng.standard_normal(size)]
    relu = np.abs(rng.standard_normal(size)) * (rng.random(size) < 0.4)
    x += [relu, -relu, np.zeros(size)]
    x.append(rng.integers(-1, 3, size).astype(np.float64))               # few distinct values
    for share in (0.03, 0.1, 0.3, 0.7):                                  # so many of them in one bucket, around the best split
        near = 0.61 + rng.integers(0, 1 << 12, size) * 2.0 ** -23
        x.append(np.where(rng.random(size) < share, near, np.abs(rng.standard_normal(size))))
    x.append(np.full(size, 8388607.0 / 4194304.0))                       # every mantissa bit set
    x.append(rng.standard_normal(size) * 2.0 ** (-30.0 * rng.random(size)))
    x.append(rng.standard_normal(size) * 1e-13)                          # below the coder's magnitudes
    x.append(rng.standard_normal(size))
    x[-1][C - 1, H - 1, W - 1] = np.nan
    x = np.stack(x).astype(np.float32)
    x[0, C // 2, 0, 0] = -0.0
    return x


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_patches_at_the_edges(case):
    import paper_1804_02941_b200 as dab
    oracle.set_threads(16)
    C, H, W, kh, kw, stride, pad = case
    x = _images(np.random.default_rng(sum(case)), C, H, W)
    desc = dab.make_desc(x.shape, 4, kh, kw, (stride, stride), (pad, pad))
    ho, wo = dab.dab_conv_output_size(desc)
    P, n = x.shape[0] * ho * wo, C * kh * kw
    new = lambda *s, dtype=torch.int32: torch.full(s, -7, dtype=dtype, device="cuda")
    c = dab.Coded(new(P, dab.dab_default_ld(n) + 4), new(P), new(P, dtype=torch.float32), new(P, dtype=torch.float32), new(P), n)
    dab.dab_set_patch_coder(dab.PATCHES_PIXEL)
    try:
        dab.dab_binarize_patches(desc, to_dev(x), c.K, c.alpha, c.beta, c.mask, c.flags)
    finally:
        dab.dab_set_patch_coder(dab.PATCHES_AUTO)
    torch.cuda.synchronize()
    check_coded(c, oracle.binarize(oracle.im2col(x, kh, kw, (stride, stride), (pad, pad))), n, log=print)
