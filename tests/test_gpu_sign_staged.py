"""Sign coding of patches by the coder that takes a warp per patch: few channels, wide windows (also wider than 32 columns), strides and
small layers, which go there, and the same shapes at batch sizes that do not; zeros of either sign and values that are not finite.
K, masks and flags bit for bit, scales within 1e-5 relative."""
import numpy as np
import pytest
import torch

import oracle
import test_gpu_sign_tiles
from parity_util import check_coded, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 33])
@pytest.mark.parametrize("C,H,W,kh,kw,stride,pad", [(3, 40, 37, 11, 11, 4, 5), (1, 28, 28, 5, 5, 1, 2), (2, 50, 49, 31, 31, 5, 0),
                                                   (2, 20, 60, 9, 33, 2, 1), (300, 5, 4, 1, 1, 1, 0), (1024, 2, 3, 1, 1, 1, 0),
                                                   (17, 9, 9, 2, 2, 1, 1), (16, 30, 31, 7, 7, 2, 3), (1, 70, 64, 64, 64, 8, 0), (33, 12, 13, 3, 3, 1, 1)])
def test_patches(C, H, W, kh, kw, stride, pad, N):
    import paper_1804_02941_b200 as dab
    oracle.set_threads(16)
    rng = np.random.default_rng(C + H + kw)
    x = rng.standard_normal((N, C, H, W)).astype(np.float32)
    x[0, 0, 0, :3] = [0.0, -0.0, -1.0]
    x[N - 1, C - 1, H - 1, W - 1] = np.inf
    n = C * kh * kw
    desc = dab.make_desc(x.shape, 4, kh, kw, (stride, stride), (pad, pad))
    ho, wo = dab.dab_conv_output_size(desc)
    P = N * ho * wo
    new = lambda *s, dtype=torch.int32: torch.full(s, -7, dtype=dtype, device="cuda")
    c = dab.Coded(new(P, dab.dab_default_ld(n) + 4), new(P), new(P, dtype=torch.float32), new(P, dtype=torch.float32), new(P), n)
    dab.dab_sign_patches(desc, to_dev(x), c.K, c.alpha, c.beta, c.mask, c.flags)
    torch.cuda.synchronize()
    check_coded(c, oracle.sign_code(oracle.im2col(x, kh, kw, (stride, stride), (pad, pad))), n, log=print)


@pytest.mark.parametrize("case", test_gpu_sign_tiles.CASES, ids=lambda c: "x".join(map(str, c)))
def test_tiles_at_batch_sizes_that_fill_them(case):
    """The edge cases of the coder by tiles, their images so many times over that they go there."""
    import paper_1804_02941_b200 as dab
    N, C, H, W, kh, kw, stride, pad = case
    rng = np.random.default_rng(sum(case) + 1)
    x = rng.standard_normal((N, C, H, W)).astype(np.float32)
    x[rng.random(x.shape) < 0.2] = 0.0
    x[rng.random(x.shape) < 0.05] = -0.0
    x[0, C - 1, H - 1, W - 1] = np.nan
    x[0, 0, 0, 0] = np.inf
    copies, n = 400, C * kh * kw
    desc = dab.make_desc((copies * N, C, H, W), 4, kh, kw, (stride, stride), (pad, pad))
    ho, wo = dab.dab_conv_output_size(desc)
    P = N * ho * wo
    new = lambda *s, dtype=torch.int32: torch.full(s, -7, dtype=dtype, device="cuda")
    c = dab.Coded(new(copies * P, dab.dab_default_ld(n)), new(copies * P), new(copies * P, dtype=torch.float32),
                  new(copies * P, dtype=torch.float32), new(copies * P), n)
    dab.dab_sign_patches(desc, to_dev(x).repeat(copies, 1, 1, 1), c.K, c.alpha, c.beta, c.mask, c.flags)
    torch.cuda.synchronize()
    for t in (c.K, c.alpha, c.beta, c.mask, c.flags):
        bits = t.view(torch.int32).view(copies, P, -1)
        assert torch.equal(bits, bits[:1].expand_as(bits))
    first = dab.Coded(c.mask[:P], c.K[:P], c.alpha[:P], c.beta[:P], c.flags[:P], n)
    check_coded(first, oracle.sign_code(oracle.im2col(x, kh, kw, (stride, stride), (pad, pad))), n)
