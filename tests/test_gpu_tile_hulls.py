"""Patches that leave the tile coder more values than a warp's 32, against the CPU checker: sorted, two to 32 a lane, or marked (few are
narrowed here, see test_gpu_narrowed_hulls.py).  Heavy tails (a few dozen to a few hundred values, as in a residual network), zeros among
the values, many equal values, clusters of values too close for another bucket width, and two far clusters with nearly the same
objective."""
import numpy as np
import pytest
import torch

import oracle
from parity_util import check_coded, to_dev

pytestmark = pytest.mark.gpu

CASES = [  # C, H, W, kh, kw, stride, pad
    (64, 15, 17, 3, 3, 1, 1),    # n = 576: what cannot be narrowed is marked
    (128, 9, 10, 3, 3, 2, 1),    # n = 1152: sorted
    (200, 7, 8, 3, 3, 1, 1),     # n = 1800: 64 buckets, sorted
    (300, 5, 6, 3, 3, 1, 0),     # channels in 16 bits
    (24, 11, 12, 5, 5, 1, 2),    # other windows: sorted
    (40, 9, 9, 2, 4, 1, 0),
    (30, 9, 12, 6, 7, 1, 3),     # two pixels per lane
    (85, 9, 11, 3, 3, 1, 1),     # n = 765 and 774: on either side of what is marked and sorted
    (86, 9, 11, 3, 3, 1, 1),
    (170, 8, 7, 3, 3, 1, 0),     # n = 1530
]


def _images(rng, C, H, W):
    size = (C, H, W)
    normal = rng.standard_normal(size)
    x = [normal * np.abs(normal), np.exp(2.0 * normal), np.abs(normal) ** 3 - 0.4]
    x.append(np.where(rng.random(size) < 0.5, x[0], 0.0))                              # zeros in the middle
    x.append(np.round(x[0] * 16.0) / 16.0)                                             # many equal ones
    x.append(np.where(rng.random(size) < 0.3, 0.75 + rng.integers(0, 200, size) * 2.0 ** -24, x[0]))
    x.append(np.where(rng.random(size) < 0.5, 1.0, -1.0) + 0.3 * rng.standard_normal(size) ** 3)
    x.append(100.0 + rng.standard_normal(size))                                        # all of one bucket or two
    x.append(rng.standard_normal(size) * 4.0 ** rng.integers(-4, 5, (C, 1, 1)))        # channels of unlike scale
    return np.stack(x).astype(np.float32)


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_long_hulls(case):
    import paper_1804_02941_b200 as dab
    oracle.set_threads(16)
    C, H, W, kh, kw, stride, pad = case
    x = _images(np.random.default_rng(sum(case)), C, H, W)
    desc = dab.make_desc(x.shape, 4, kh, kw, (stride, stride), (pad, pad))
    ho, wo = dab.dab_conv_output_size(desc)
    P, n = x.shape[0] * ho * wo, C * kh * kw
    new = lambda *s, dtype=torch.int32: torch.full(s, -7, dtype=dtype, device="cuda")
    c = dab.Coded(new(P, dab.dab_default_ld(n)), new(P), new(P, dtype=torch.float32), new(P, dtype=torch.float32), new(P), n)
    dab.dab_set_patch_coder(dab.PATCHES_PIXEL)
    try:
        dab.dab_binarize_patches(desc, to_dev(x), c.K, c.alpha, c.beta, c.mask, c.flags)
    finally:
        dab.dab_set_patch_coder(dab.PATCHES_AUTO)
    torch.cuda.synchronize()
    check_coded(c, oracle.binarize(oracle.im2col(x, kh, kw, (stride, stride), (pad, pad))), n, log=print)
