"""Patches that leave the tile coder 128 values and more, in 3 x 3 windows of short rows, against the CPU checker: these are narrowed to a
few before they are searched.  The bucket grid of a tile suits its average patch, so the images mix patches of unlike scale and offset.
Counted in the kernel: of 2604 patches 14 to 1475 leave that many, most of them can be narrowed (of those with many equal values less than
half), and some keep 32 to 63 values, have zeros among what is kept, or lie beside zeros and other values that are not kept.  Rows of 576
and 765 values, whose other hulls are left to the kernel for marked patches, and of 774 and 1530, whose are sorted; with a
stride also rows of 1152 and, in a layer where 32 buckets let two tiles share an SM, of 3456 values with channels in 16 bits."""
import numpy as np
import pytest
import torch

import oracle
from parity_util import check_coded, to_dev

pytestmark = pytest.mark.gpu

KINDS = ["scales", "scales0", "offsets", "heavy", "steps", "mixed"]
LAYERS = [(64, 28, 31, 3, 1), (85, 28, 31, 3, 1), (86, 28, 31, 3, 1), (170, 28, 31, 3, 1), (128, 28, 31, 3, 2), (384, 15, 15, 32, 2)]  # C, H, W, images, stride


def _image(kind, rng, C, H, W):
    n = rng.standard_normal((C, H, W))
    scale = 2.0 ** rng.integers(-6, 1, (1, (H + 6) // 7, (W + 6) // 7)).repeat(7, 1).repeat(7, 2)[:, :H, :W]
    if kind == "scales":                       # both signs, no zeros: the best split is near zero
        return n * scale
    if kind == "scales0":                      # and a third of zeros
        return n * scale * (rng.random((C, H, W)) < 0.66)
    if kind == "offsets":                      # one sign, a few octaves
        return np.abs(n * scale + 4.0 * scale)
    if kind == "heavy":
        return n * np.abs(n)
    if kind == "steps":                        # many equal values
        return np.round(n * 32.0 * scale) / 8.0
    return np.where(rng.random((C, H, W)) < 0.5, n * scale, (np.abs(n) + 3.0) * scale)


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("C,H,W,images,stride", LAYERS)
def test_narrowed_hulls(kind, C, H, W, images, stride):
    import paper_1804_02941_b200 as dab
    oracle.set_threads(16)
    rng = np.random.default_rng(C)
    x = np.stack([_image(kind, rng, C, H, W) for _ in range(images)]).astype(np.float32)
    desc = dab.make_desc(x.shape, 4, 3, 3, (stride, stride), (1, 1))
    ho, wo = dab.dab_conv_output_size(desc)
    P, n = x.shape[0] * ho * wo, C * 9
    new = lambda *s, dtype=torch.int32: torch.full(s, -7, dtype=dtype, device="cuda")
    c = dab.Coded(new(P, dab.dab_default_ld(n)), new(P), new(P, dtype=torch.float32), new(P, dtype=torch.float32), new(P), n)
    dab.dab_set_patch_coder(dab.PATCHES_PIXEL)
    try:
        dab.dab_binarize_patches(desc, to_dev(x), c.K, c.alpha, c.beta, c.mask, c.flags)
    finally:
        dab.dab_set_patch_coder(dab.PATCHES_AUTO)
    torch.cuda.synchronize()
    check_coded(c, oracle.binarize(oracle.im2col(x, 3, 3, (stride, stride), (1, 1))), n, log=print)
