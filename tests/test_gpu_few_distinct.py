"""Rows of few distinct values, whose hull no bucket grid takes apart: the table of distinct values of the CTA-per-row coder at the
numbers it changes at (a warp's 32, its capacities of 96, 192 and 256 by row length) and beyond, with and without zeros, of one
sign and both, outside the magnitudes the grid resolves, and beside many other values.  Against the CPU checker; in integers and
few bits, so that exact ties occur and the rule for them decides."""
import numpy as np
import pytest
import torch

import oracle
from parity_util import check_coded, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,cap", [(300, 96), (1024, 96), (1025, 192), (4096, 192), (4097, 256), (16384, 256)])
def test_rows_of_few_distinct_values(n, cap):
    import paper_1804_02941_b200 as dab
    oracle.set_threads(16)
    rng = np.random.default_rng(n)
    rows = []
    for k in (1, 2, 3, 31, 32, 33, cap - 1, cap, cap + 1, 2 * cap):
        values = (1.0 + np.arange(k) / 1024.0) * 0.75                   # within an octave
        rows.append(values[rng.integers(0, k, n)])
        rows.append(-values[rng.integers(0, k, n)] * (rng.random(n) < 0.7))   # the other sign, with zeros
        spread = (np.arange(k) - k // 2) * 0.25                        # both signs, zero among them
        rows.append(spread[rng.integers(0, k, n)])
        rows.append(spread[rng.integers(0, k, n)] * 1e20)              # beyond the grid's magnitudes
        rows.append(spread[rng.integers(0, k, n)] * 1e-30)
    pm = np.ones(n)
    pm[: n // 2] = -1.0                                                # halves of +1 and -1: every split between them ties
    rows += [pm, np.sign(rng.standard_normal(n)), np.zeros(n)]
    near = rng.standard_normal(n)                                      # one value holds two thirds of a row
    near[rng.random(n) < 0.67] = 0.61
    rows.append(near)
    w = np.stack(rows).astype(np.float32)
    w[1, 0] = -0.0
    got = dab.dab_binarize(to_dev(w))
    torch.cuda.synchronize()
    check_coded(got, oracle.binarize(w), n, log=print)


@pytest.mark.parametrize("C,k", [(64, 3), (96, 5), (600, 3)])
def test_patches_of_few_distinct_values(C, k):
    import paper_1804_02941_b200 as dab
    oracle.set_threads(16)
    rng = np.random.default_rng(C)
    shape = (C, 9, 8)
    x = np.stack([np.sign(rng.standard_normal(shape)), rng.integers(-1, 2, shape), rng.random(shape) < 0.3,
                  np.full(shape, 0.5), np.round(np.abs(rng.standard_normal(shape)) * 4) / 4,
                  np.where(rng.random(shape) < 0.8, 0.61, rng.standard_normal(shape))]).astype(np.float32)
    n = C * k * k
    desc = dab.make_desc(x.shape, 4, k, k, (1, 1), (k // 2, k // 2))
    P = x.shape[0] * 72
    new = lambda *s, dtype=torch.int32: torch.full(s, -7, dtype=dtype, device="cuda")
    for coder in (dab.PATCHES_PIXEL, dab.PATCHES_AUTO):
        c = dab.Coded(new(P, dab.dab_default_ld(n)), new(P), new(P, dtype=torch.float32), new(P, dtype=torch.float32), new(P), n)
        dab.dab_set_patch_coder(coder)
        try:
            dab.dab_binarize_patches(desc, to_dev(x), c.K, c.alpha, c.beta, c.mask, c.flags)
        finally:
            dab.dab_set_patch_coder(dab.PATCHES_AUTO)
        torch.cuda.synchronize()
        check_coded(c, oracle.binarize(oracle.im2col(x, k, k, (1, 1), (k // 2, k // 2))), n, log=print)
