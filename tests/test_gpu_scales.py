"""Contraction with scales that no coder writes: the contraction calls take any values of the set and the clear bits, and an
output is the sum of the four terms, also where some of them are empty and the values differ by many orders of magnitude.

The reference forms the four terms in fp64 in the order of the header, each operation rounded, and rounds once to fp32: the
outputs are compared bit for bit (NaN for NaN), except where both rows are ordered as the coders' are (the set bits' value no
smaller in magnitude): those may be gathered, which is good to 2^-49 of the terms' magnitudes before the rounding to fp32.
Shapes reach every kernel and both output layouts, which agree to the bit."""
import numpy as np
import pytest
import torch

from parity_util import to_dev

pytestmark = pytest.mark.gpu


def masks(rng, rows, n, subset_of=None):
    e = rng.random((rows, n)) < rng.random((rows, 1))
    if subset_of is not None:
        e &= subset_of
    e[0] = subset_of if subset_of is not None else True   # a full row: its clear bits' terms are empty
    return e


def scales(rng, rows):
    """(value of the set bits, value of the clear bits): of very different size, either way round, zeros and infinities."""
    a = (rng.standard_normal(rows) * 10.0 ** rng.integers(-12, 13, rows)).astype(np.float32)
    b = (rng.standard_normal(rows) * 10.0 ** rng.integers(-12, 13, rows)).astype(np.float32)
    a[::7] = 0.0
    b[3::7] = 0.0
    a[-1:] = np.inf
    return a, b


def four_terms(e, f, alpha, beta, gamma, delta):
    n = e.shape[1]
    p11 = f.astype(np.float32) @ e.astype(np.float32).T   # counts below 2^24: exact
    p11 = p11.astype(np.float64)
    Ke, Kf = e.sum(1).astype(np.float64)[None, :], f.sum(1).astype(np.float64)[:, None]
    a, b, g, d = (v.astype(np.float64) for v in (alpha, beta, gamma, delta))
    with np.errstate(all="ignore"):
        y = (a[None, :] * g[:, None]) * p11
        y = y + (a[None, :] * d[:, None]) * (Ke - p11)
        y = y + (b[None, :] * g[:, None]) * (Kf - p11)
        y = y + (b[None, :] * d[:, None]) * (n - Ke - Kf + p11)
        size = (np.abs(a) * np.abs(g[:, None])) * p11 + (np.abs(a) * np.abs(d[:, None])) * (Ke - p11) \
            + (np.abs(b) * np.abs(g[:, None])) * (Kf - p11) + (np.abs(b) * np.abs(d[:, None])) * (n - Ke - Kf + p11)
        ordered = ((np.abs(a) >= np.abs(b)) & np.isfinite(a))[None, :] & ((np.abs(g) >= np.abs(d)) & np.isfinite(g))[:, None]
        slack = np.where(ordered, 2.0 ** -23 * np.abs(y) + 2.0 ** -49 * size, 0.0)
        return y.astype(np.float32), slack, p11.astype(np.int32)


def same(got, ref, slack):
    with np.errstate(all="ignore"):
        near = np.abs(got.astype(np.float64) - ref.astype(np.float64)) <= slack
    return ((got == ref) | (np.isnan(got) & np.isnan(ref)) | near).all()


# one tile, ragged; narrow and wide column tiles; 182 tiles of long rows; few rows (split over clusters when forced)
@pytest.mark.parametrize("M,N,n", [(16, 40, 130), (150, 70, 300), (300, 513, 2304), (1700, 1601, 1100), (9, 100, 4000)])
def test_any_scales(M, N, n):
    import paper_1804_02941_b200 as dab
    rng = np.random.default_rng(M + n)
    base = rng.random(n) < 0.5
    f, e = masks(rng, M, n, base), masks(rng, N, n, base)
    f[M // 2:] |= rng.random((M - M // 2, n)) < 0.3
    gamma, delta = scales(rng, M)
    alpha, beta = scales(rng, N)
    ref, slack, refP = four_terms(e, f, alpha, beta, gamma, delta)

    def coded(bits, v1, v0):
        mask, K = dab.dab_pack(to_dev(bits.astype(np.uint8)))
        return dab.Coded(mask, K, to_dev(v1), to_dev(v0), torch.zeros_like(K), n)
    a, b = coded(f, gamma, delta), coded(e, alpha, beta)
    desc = dab.make_desc((M, n, 1, 1), N, 1, 1)
    y = torch.empty((M, N, 1, 1), device="cuda")
    out = {}
    for path in (dab.CONTRACT_TENSOR, dab.CONTRACT_POPC):
        dab.dab_set_contraction(path)
        try:
            got, p11 = dab.dab_binary_gemm(a, b, want_p11=True)
            dab.dab_binary_conv_contract(desc, a.mask, a.K, a.alpha, a.beta, b, y)
        finally:
            dab.dab_set_contraction(dab.CONTRACT_AUTO)
        torch.cuda.synchronize()
        assert np.array_equal(p11.cpu().numpy(), refP)
        assert same(got.cpu().numpy(), ref, slack)
        assert torch.equal(y.view(M, N).view(torch.int32), got.view(torch.int32))
        out[path] = got
    assert torch.equal(out[dab.CONTRACT_TENSOR].view(torch.int32), out[dab.CONTRACT_POPC].view(torch.int32))
