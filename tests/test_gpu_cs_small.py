"""CountSketch of small dense A: the gather takes little more than the short
kernels before it, as it does with enough teams for its rows and buckets."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,r", [(2_000, 36, 4_000), (1_500, 256, 3_000)])
def test_gather_beside_the_sort(n, d, r):
    import paper_2203_02798_gb300 as lsk
    A = torch.randn((n, d), generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")
    for _ in range(3):
        lsk.cs_sketch(A, r, 1)
    ctx = lsk.context()
    ratios = []
    for _ in range(5):
        ctx.profile_reset()
        ctx.profile(True)
        for _ in range(30):
            lsk.cs_sketch(A, r, 1)
        ctx.sync()
        ms = {k: v[1] for k, v in ctx.profile_totals().items()}
        ctx.profile(False)
        ratios.append(3 * ms["cs_dense_gather"] / (ms["cs_count"] + ms["cs_scan"] + ms["cs_place"]))
    assert sorted(ratios)[2] <= 1.42


# a bucket a team, two, several; rows fewer and more than buckets; the last ones of each
@pytest.mark.parametrize("n,d,r", [(1, 8, 1), (3, 33, 5), (1_000, 32, 1_000), (1_000, 32, 999), (4_863, 40, 4_864),
                                   (10_000, 50, 4_865), (3_000, 100, 9_729), (7_999, 36, 1_000), (8_001, 36, 1_000),
                                   (40_000, 256, 30_000), (2_000, 31, 4_863)])
def test_whole_numbers_are_summed_exactly(n, d, r):
    import paper_2203_02798_gb300 as lsk
    g = torch.Generator(device="cuda").manual_seed(d)
    A = torch.randint(-50, 51, (n, d), generator=g, device="cuda").float()
    h, s = lsk.debug_hash(n, r, 5)
    want = torch.zeros((r, d), device="cuda")
    want.index_add_(0, h.long(), A * s.float()[:, None])
    assert torch.equal(lsk.cs_sketch(A, r, 5), want)
