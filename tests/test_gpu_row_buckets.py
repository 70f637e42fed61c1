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


@pytest.mark.parametrize("case", [  # N, C, H, W, kh, kw, stride, pad: layers of fewer than 1024 patches, or long ones
    (2, 29, 9, 7, 3, 3, 1, 1),      # n = 261: the shortest of the path, padding
    (1, 115, 6, 8, 3, 3, 2, 0),     # n = 1035
    (3, 40, 5, 6, 2, 3, 1, 2),      # n = 240 takes the warp kernel; windows in the padding alone
    (1, 456, 5, 5, 3, 3, 1, 1),     # n = 4104
    (2, 1025, 3, 3, 3, 3, 1, 0),    # n = 9225, fully connected, unaligned rows
    (5, 130, 2, 2, 2, 2, 1, 0),     # n = 520, fully connected, aligned
    (1, 1300, 3, 2, 1, 1, 1, 0),    # 1 x 1 windows
    (1, 200, 12, 11, 7, 7, 1, 3),   # n = 9800, more than 8192 values
], ids=lambda c: "x".join(map(str, c)))
@pytest.mark.parametrize("signed", [False, True])
def test_small_layers(case, signed):
    import paper_1804_02941_b200 as dab
    oracle.set_threads(16)
    N, C, H, W, kh, kw, stride, pad = case
    rng = np.random.default_rng(sum(case))
    x = rng.standard_normal((N, C, H, W))
    if not signed:
        x = np.abs(x) * (rng.random(x.shape) < 0.4)
    x = x.astype(np.float32)
    desc = dab.make_desc(x.shape, 4, kh, kw, (stride, stride), (pad, pad))
    ho, wo = dab.dab_conv_output_size(desc)
    P, n = N * ho * wo, C * kh * kw
    new = lambda *s, dtype=torch.int32: torch.full(s, -7, dtype=dtype, device="cuda")
    c = dab.Coded(new(P, dab.dab_default_ld(n)), new(P), new(P, dtype=torch.float32), new(P, dtype=torch.float32), new(P), n)
    dab.dab_binarize_patches(desc, to_dev(x), c.K, c.alpha, c.beta, c.mask, c.flags)
    torch.cuda.synchronize()
    check_coded(c, oracle.binarize(oracle.im2col(x, kh, kw, (stride, stride), (pad, pad))), n, log=print)
