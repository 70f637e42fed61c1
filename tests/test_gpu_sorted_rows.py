"""Rows whose hull is too long for the CTA-per-row coder and whose values are too many to count: every warp of the CTA looks at a
sample of the staged values before these are sorted in place.  Many rows at every row length of the coder, in matrices and as filters
of a training step, against the checker and the same at every run."""
import numpy as np
import pytest
import torch

import oracle
from parity_util import check_coded, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,rows", [(300, 4096), (700, 2048), (1024, 2048), (2304, 1024), (4096, 512), (9216, 256)])
def test_rows_of_many_close_values(n, rows):
    import paper_1804_02941_b200 as dab
    oracle.set_threads(16)
    rng = np.random.default_rng(n)
    w = 1.0 + rng.random((rows, n)) / 32.0                                  # one bucket holds a row
    w[1::2] *= rng.choice([-1.0, 1.0], (rows // 2, 1))
    w[::4, : n // 3] = -2.0 * w[::4, : n // 3]                               # or two rows of it on either side of zero
    w = w.astype(np.float32)
    wd = to_dev(w)
    first = dab.dab_binarize(wd)
    fields = ("mask", "K", "alpha", "beta", "flags")
    for _ in range(20):
        again = dab.dab_binarize(wd)
        for f in fields:
            assert torch.equal(getattr(first, f).view(torch.int32), getattr(again, f).view(torch.int32)), f
    _, coded, _ = dab.dab_binarize_train(wd - 1.0)
    _, again, _ = dab.dab_binarize_train(wd - 1.0)
    for f in fields:
        assert torch.equal(getattr(coded, f).view(torch.int32), getattr(again, f).view(torch.int32)), f
    torch.cuda.synchronize()
    check_coded(first, oracle.binarize(w), n, log=print)
