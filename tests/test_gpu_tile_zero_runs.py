"""Patches with a run of exact zeros and two splits of nearly the same objective, one beside the zeros and one far from them, through
the tile coder and against the CPU checker: the values left after pruning then reach from one split to the other, with the zeros
among them, and narrowing them must not lose the better one.  Every patch is an image of its own (3 x 3 windows, no padding)."""
import numpy as np
import pytest
import torch

import oracle
from parity_util import check_coded, to_dev

pytestmark = pytest.mark.gpu


def _objective(v):
    v = np.sort(v.astype(np.float64))
    P, s, n = np.cumsum(v)[:-1], np.arange(1, v.size), v.size
    return P * P / s + (v.sum() - P) ** 2 / (n - s)


def _patch(far, far_at, middle, small, zeros, high, high_at, n):
    i = np.arange
    v = [-far_at * (1 + i(far) / 64), -(1 + i(middle) / 512), -(0.5 + i(small) / 512), np.zeros(zeros), high_at * (1 + i(high) / 1024)]
    return np.concatenate(v).astype(np.float32)


def _tied(rng, n):
    """far_at such that the split behind the `far` values and the best one from the small values on agree to some 1e-5."""
    while True:
        far, middle, small, zeros = (int(rng.integers(*r)) for r in ((3, 30), (40, 150), (1, 40), (1, 80)))
        high, high_at = n - far - middle - small - zeros, rng.uniform(0.9, 1.7)
        lo, hi = 1.5, 40.0
        for _ in range(40):
            mid = 0.5 * (lo + hi)
            D = _objective(_patch(far, mid, middle, small, zeros, high, high_at, n))
            if D[:far].max() > D[far + middle - 1:].max():
                hi = mid
            else:
                lo = mid
        if lo > 1.6 and hi < 39.0:
            return _patch(far, lo * (1 + rng.uniform(-3e-5, 3e-5)), middle, small, zeros, high, high_at, n)


@pytest.mark.parametrize("C", [64, 112])   # rows of 576 and 1008 values
def test_splits_beside_the_zeros_and_far_from_them(C):
    import paper_1804_02941_b200 as dab
    oracle.set_threads(16)
    rng, n = np.random.default_rng(C), 9 * C
    rows = [_tied(rng, n) for _ in range(1000)]
    if C == 64:   # splits 9 (objective 1309.226) and 108 (1309.298)
        rows.append(_patch(9, 8.349121094, 89, 10, 21, 447, 1.259277344, n))
    rows = np.stack(rows)
    rows = np.stack([r[rng.permutation(n)] for r in np.concatenate([rows, -rows])])
    x = rows.reshape(-1, C, 3, 3)
    desc = dab.make_desc(x.shape, 4, 3, 3, (1, 1), (0, 0))
    new = lambda *s, dtype=torch.int32: torch.full(s, -7, dtype=dtype, device="cuda")
    P = len(x)
    c = dab.Coded(new(P, dab.dab_default_ld(n)), new(P), new(P, dtype=torch.float32), new(P, dtype=torch.float32), new(P), n)
    dab.dab_set_patch_coder(dab.PATCHES_PIXEL)
    try:
        dab.dab_binarize_patches(desc, to_dev(x), c.K, c.alpha, c.beta, c.mask, c.flags)
    finally:
        dab.dab_set_patch_coder(dab.PATCHES_AUTO)
    torch.cuda.synchronize()
    check_coded(c, oracle.binarize(rows), n, log=print)
