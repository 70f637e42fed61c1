"""The tile coder where the images are many and small, so that a tile holds a whole one: pixels on either side of where the way
of summing a pixel's buckets changes (80), with one and two buckets per lane.  The same images again and again: the first are
compared with the CPU checker, the others with the first."""
import numpy as np
import pytest
import torch

import oracle
from parity_util import check_coded, to_dev
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
