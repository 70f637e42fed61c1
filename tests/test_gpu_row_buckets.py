"""The CTA-per-row coder of dab_binarize at the edges of its row-length ranges, against the CPU checker: lengths around
the changes of CTA size, unaligned rows (scalar staging), hulls that no bucket separates (few distinct values, one
bucket holding the row: the in-place sort), values below the resolved octaves, constant, zero and non-finite rows."""
import numpy as np
import pytest
import torch

import oracle
from parity_util import check_coded, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("aligned", [True, False])
@pytest.mark.parametrize("n", [257, 1023, 1024, 1025, 2300, 4095, 4096, 4097, 9216, 12545, 16384])
def test_rows_at_the_edges(n, aligned):
    import paper_1804_02941_b200 as dab
    oracle.set_threads(16)
    rng = np.random.default_rng(n)
    w = rng.standard_normal((14, n))
    w[1] = np.abs(w[1]) * (rng.random(n) < 0.4)           # post-ReLU
    w[2] = -w[1]                                          # one sign, the other one
    w[3] = rng.integers(0, 3, n)                          # three distinct values: every one a bucket of its own
    w[4] = 1.0 + rng.integers(0, 64, n) * 2.0 ** -23      # one bucket
    w[5] = 2.5                                            # constant
    w[6] = 0.0
    w[7, rng.integers(0, n)] = np.nan
    w[8, 0] = 5e4                                         # almost everything below the resolved octaves
    w[9] = w[9] * 2.0 ** (-30.0 * rng.random(n))
    w[10] = np.where(rng.random(n) < 0.9, 1e-3, 1.0) * np.sign(w[10])
    w[11] = w[11] * 1e20                                  # outside the magnitude window
    w[12] = 0.0
    w[12, n - 1] = -1.0                                   # one value
    w = w.astype(np.float32)
    base = torch.zeros((14, n + (7 if not aligned else (-n) % 4)), device="cuda")
    rows = base[:, 3:3 + n] if not aligned else base[:, :n]
    rows.copy_(to_dev(w))
    got = dab.dab_binarize(rows)
    torch.cuda.synchronize()
    check_coded(got, oracle.binarize(w), n, log=print)
