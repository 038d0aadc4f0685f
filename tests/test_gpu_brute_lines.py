"""Where the exact search goes to the tensor cores: the sizes at which one warp per
query measured faster stay there (one launch), the others give the oracle's answer
on the tensor cores (a second launch looks for rows given up) on both sides of the
line, for every row width and list length that has a line of its own."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def search(db, q, k):
    from oracle import oracle as O
    from paper_1209_0410_gb300 import hc
    before = hc.hc_launch_count()
    ids, dist = hc.hc_bruteforce(torch.from_numpy(db).cuda(), torch.from_numpy(q).cuda(), k)
    launches = hc.hc_launch_count() - before
    rids, rdist = O.bruteforce(db, q, k)
    assert np.array_equal(ids.cpu().numpy(), rids)
    assert np.array_equal(dist.cpu().numpy(), O.int32_dist(rdist))
    return launches


@pytest.mark.parametrize("d,n,k", [(16, 4096, 10), (64, 4096, 16), (64, 8192, 10), (48, 12_288, 16),
                                   (64, 32_768, 112), (32, 49_152, 100), (128, 4096, 16),
                                   (96, 32_768, 112)])
def test_one_warp_per_query_where_it_is_faster(d, n, k):
    rng = np.random.default_rng(n + k)
    db = rng.integers(0, 256, (n, d), dtype=np.uint8)
    assert search(db, rng.integers(0, 256, (40, d), dtype=np.uint8), k) == 1


@pytest.mark.parametrize("d,line,k", [
    (16, 6450, 1), (48, 10_250, 5), (64, 15_000, 10), (32, 20_700, 16), (64, 32_768, 17),
    (16, 32_768, 48), (64, 34_375, 80), (48, 58_928, 100), (64, 103_125, 112), (80, 6000, 11),
    (128, 6000, 16), (128, 4096, 10), (128, 47_500, 112), (256, 4096, 16), (256, 32_768, 48)])
def test_both_sides_of_a_line(d, line, k):
    rng = np.random.default_rng(line + d)
    db = rng.integers(0, 256, (line, d), dtype=np.uint8)
    q = rng.integers(0, 256, (33, d), dtype=np.uint8)
    assert search(db[:line - 1], q, k) == 1
    assert search(db, q, k) > 1
