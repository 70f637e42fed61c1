"""The same input gives the same bits at every run, whatever order the threads of a tile come in: patches whose values lie below
the octaves that the tile coder's grid resolves (a few pixels of 1.0 are in every tile), one larger value in each, pairs that
cancel and a rest far below them: the mean of all but the largest is what an fp64 sum of them rounds away or keeps."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _same_codes_every_run(dab, x, g):
    w = dab.dab_binarize(torch.randn((16, x.shape[1] * 9), device="cuda", generator=g))
    dab.dab_set_patch_coder(dab.PATCHES_PIXEL)
    try:
        first = None
        for _ in range(40):
            y, d = dab.dab_binary_conv(x, w, 3, 3, (1, 1), (1, 1), details=True)
            bits = [t.view(torch.int32).clone() for t in (d.pK, d.pgamma, d.pdelta, d.pmask, y)]
            first = first or bits
            for name, now, then in zip(("K", "gamma", "delta", "mask", "y"), bits, first):
                assert torch.equal(now, then), "%s differs between runs" % name
    finally:
        dab.dab_set_patch_coder(dab.PATCHES_AUTO)


@pytest.mark.parametrize("C,low", [(64, 2.0 ** -9), (256, 2.0 ** -13)])   # 8 and 12 resolved octaves
@pytest.mark.parametrize("anchor", [0.0, 2.0])   # 2: every patch has a value of the lowest resolved octave as well
def test_sums_of_unresolved_values_do_not_depend_on_the_order(C, low, anchor):
    import paper_1804_02941_b200 as dab
    g = torch.Generator(device="cuda")
    g.manual_seed(C)

    def uniform(*shape):
        return torch.rand(shape, device="cuda", generator=g)
    k = C // 4
    pair = low * 2.0 ** -3 * (1.0 + uniform(8, k, 28, 28))
    rest = low * 2.0 ** -36 * (uniform(8, 2 * k, 28, 28) - 0.4)
    x = torch.cat([pair, -pair, rest], dim=1)[:, torch.randperm(C, generator=torch.Generator().manual_seed(1)).cuda()].contiguous()
    x[:, 5] = torch.where(uniform(8, 28, 28) < 0.2, low * 0.99, 0.0)
    if anchor:
        x[:, 7] = anchor * low
    x[:, 6, ::4, ::4] = 1.0
    _same_codes_every_run(dab, x, g)


@pytest.mark.parametrize("C", [64, 96])   # rows of 576 and 864 values
def test_sums_below_a_narrowed_search_do_not_depend_on_the_order(C):
    # a third of the values near 1, the rest far below in pairs that cancel (their negative halves lie below what is searched, their
    # positive ones are searched) and 36 octaves smaller: the mean of the low side is what is left of them
    import paper_1804_02941_b200 as dab
    g = torch.Generator(device="cuda")
    g.manual_seed(C)

    def uniform(*shape):
        return torch.rand(shape, device="cuda", generator=g)
    k = C // 5
    pair = 2.0 ** -10 * (1.0 + uniform(8, k, 28, 28))
    rest = 2.0 ** -45 * uniform(8, k, 28, 28)
    high = 0.7 + 0.3 * uniform(8, C - 3 * k, 28, 28)
    x = torch.cat([pair, -pair, rest, high], dim=1)[:, torch.randperm(C, generator=torch.Generator().manual_seed(1)).cuda()].contiguous()
    _same_codes_every_run(dab, x, g)
