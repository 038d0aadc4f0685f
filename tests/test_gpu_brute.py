"""Exact search on the tensor cores (uint8 rows of at most 256 bytes) against the
oracle: the edges of the query tiles (128, 256), the row tiles (32, 64, 128) and
the cluster's shares, every list width, and the largest distances a row can have."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def check(db, q, k):
    from oracle import oracle as O
    from paper_1209_0410_gb300 import hc
    ids, dist = hc.hc_bruteforce(torch.from_numpy(db).cuda(), torch.from_numpy(q).cuda(), k)
    rids, rdist = O.bruteforce(db, q, k)
    assert np.array_equal(ids.cpu().numpy(), rids)
    assert np.array_equal(dist.cpu().numpy(), O.int32_dist(rdist))


@pytest.mark.parametrize("d", [16, 48, 64, 80, 128, 144, 256])
@pytest.mark.parametrize("k", [1, 10, 16, 17, 48, 49, 112, 128])
def test_widths_and_lists(d, k):
    rng = np.random.default_rng(d * 1000 + k)
    n = 4097 if k <= 16 else 32_801
    db = rng.integers(0, 256, (n, d), dtype=np.uint8)
    check(db, rng.integers(0, 256, (33, d), dtype=np.uint8), k)


@pytest.mark.parametrize("n,nq", [(4096, 1), (4223, 127), (4225, 128), (4097, 129), (8192, 256),
                                  (8191, 257), (40_001, 5), (5000, 1100), (4100, 4500)])
def test_tile_and_share_edges(n, nq):
    from paper_1209_0410_gb300 import datagen
    db = datagen.make_db(n, 128, seed=n)
    check(db, datagen.make_queries(db, nq, seed=nq), 10)


@pytest.mark.parametrize("d", [128, 256])
def test_extreme_values_and_ties(d):
    """Rows and queries of 0 and 255 only (distances up to 255^2 d) in many copies:
    every k-th distance is a tie, decided by the lower id."""
    rng = np.random.default_rng(d)
    few = (rng.integers(0, 2, (7, d)) * 255).astype(np.uint8)
    few[0], few[1] = 0, 255
    q = np.concatenate([few, 255 - few])
    check(few[rng.integers(0, 7, 5000)], q, 16)
    check(few[rng.integers(0, 7, 40_000)], q, 40)
