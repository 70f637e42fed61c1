"""The tile coder where the images are many and small, so that a tile holds a whole one: pixels on either side of where the way
of summing a pixel's buckets changes (80), with one and two buckets per lane.  The same images again and again: the first are
compared with the CPU checker, the others with the first.  And windows of more than 32 pixels, pixels of more than 512 channels."""
import numpy as np
import pytest
import torch

import oracle
from parity_util import check_coded, to_dev
import test_gpu_tile_patches
from test_gpu_tile_patches import _images

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,H,W", [(40, 7, 11), (40, 8, 10), (40, 9, 9), (171, 7, 11), (171, 8, 10)])
def test_tiles_of_whole_images(C, H, W):
    import paper_1804_02941_b200 as dab
    oracle.set_threads(16)
    x = _images(np.random.default_rng(C + H), C, H, W)
    n, images, copies = C * 9, x.shape[0], 40
    desc = dab.make_desc((copies * images, C, H, W), 4, 3, 3, (1, 1), (1, 1))
    P = copies * images * H * W
    new = lambda *s, dtype=torch.int32: torch.full(s, -7, dtype=dtype, device="cuda")
    c = dab.Coded(new(P, dab.dab_default_ld(n)), new(P), new(P, dtype=torch.float32), new(P, dtype=torch.float32), new(P), n)
    dab.dab_set_patch_coder(dab.PATCHES_PIXEL)
    try:
        dab.dab_binarize_patches(desc, to_dev(x).repeat(copies, 1, 1, 1), c.K, c.alpha, c.beta, c.mask, c.flags)
    finally:
        dab.dab_set_patch_coder(dab.PATCHES_AUTO)
    torch.cuda.synchronize()
    first = images * H * W
    for t in (c.K, c.alpha, c.beta, c.mask, c.flags):
        bits = t.view(torch.int32).view(copies, first, -1)
        assert torch.equal(bits, bits[:1].expand_as(bits))
    one = dab.Coded(c.mask[:first], c.K[:first], c.alpha[:first], c.beta[:first], c.flags[:first], n)
    check_coded(one, oracle.binarize(oracle.im2col(x, 3, 3, (1, 1), (1, 1))), n, log=print)


@pytest.mark.parametrize("case", [  # C, H, W, kh, kw, stride, pad
    (9, 14, 6, 11, 3, 1, 1),      # 33 pixels: one in the upper half of the lanes' pairs; n = 297
    (8, 9, 12, 6, 6, 1, 3),       # 36
    (40, 11, 9, 7, 7, 2, 3),      # 49, n = 1960
    (33, 8, 9, 9, 7, 1, 4),       # 63
    (128, 8, 9, 8, 8, 1, 2),      # 64, n = 8192
    (513, 4, 4, 3, 3, 1, 1),      # a pixel's bucket may hold more mantissas than 32 bits
    (910, 3, 4, 3, 3, 1, 1),      # n = 8190
    (2048, 3, 2, 2, 2, 1, 1),     # n = 8192
    (2000, 2, 3, 1, 1, 1, 0),
], ids=lambda c: "x".join(map(str, c)))
def test_wide_windows_and_many_channels(case):
    test_gpu_tile_patches.test_patches_at_the_edges(case)
