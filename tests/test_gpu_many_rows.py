"""Matrices of so many short rows that each gets one warp: the row coder at the ends of that range of lengths, on rows that the
search settles, rows that it leaves (few distinct values, magnitudes outside its window) and trivial ones.  The first rows
against the CPU checker, the same rows again further on against the first."""
import numpy as np
import pytest
import torch

import oracle
from parity_util import check_coded, to_dev

pytestmark = pytest.mark.gpu


def _rows(n):
    rng = np.random.default_rng(n)
    w = rng.standard_normal((21, n))
    w[1] = np.abs(w[1]) * (rng.random(n) < 0.4)
    w[2] = -w[1]
    w[3] = rng.integers(0, 3, n)
    w[4] = 1.0 + rng.integers(0, 64, n) * 2.0 ** -23
    w[5] = 2.5
    w[6] = 0.0
    w[7, rng.integers(0, n)] = np.nan
    w[8, 0] = 5e4
    w[9] = w[9] * 2.0 ** (-30.0 * rng.random(n))
    w[10] = np.where(rng.random(n) < 0.9, 1e-3, 1.0) * np.sign(w[10])
    w[11] = w[11] * 1e20
    w[12] = 0.0
    w[12, n - 1] = -1.0
    w[13] = np.sign(w[13])
    w[14] = np.round(np.abs(w[14]) * 4) / 4
    w[15] = rng.laplace(0.0, 0.05, n)
    w[16] = np.exp(4 * w[16])
    w[17] = np.abs(w[17])
    w[18] = -np.abs(w[18])
    w[19] = rng.integers(-200, 200, n) / 128.0
    return w.astype(np.float32)


@pytest.mark.parametrize("aligned", [True, False])
@pytest.mark.parametrize("n", [257, 300, 511, 512])
def test_a_warp_per_row(n, aligned):
    import paper_1804_02941_b200 as dab
    oracle.set_threads(16)
    w = _rows(n)
    copies = 160   # 3360 rows: 20 for every SM
    base = torch.zeros((copies * 21, n + (7 if not aligned else (-n) % 4)), device="cuda")
    rows = base[:, 3:3 + n] if not aligned else base[:, :n]
    rows.copy_(to_dev(w).repeat(copies, 1))
    got = dab.dab_binarize(rows)
    torch.cuda.synchronize()
    for t in (got.K, got.alpha, got.beta, got.mask, got.flags):
        bits = t.view(torch.int32).view(copies, 21, -1)
        assert torch.equal(bits, bits[:1].expand_as(bits))
    check_coded(dab.Coded(got.mask[:21], got.K[:21], got.alpha[:21], got.beta[:21], got.flags[:21], n), oracle.binarize(w), n, log=print)
