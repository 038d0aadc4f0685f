"""hc_probe_labels over every form of index: a label is the smallest depth whose
top-k equals the top-k at p_max, so the depths it gives reproduce that answer
and one less does not (hc_query_depths, whole numbers: no tolerance)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def rows(n, d, dtype, seed, few=0):
    from paper_1209_0410_gb300 import datagen
    db = datagen.make_db(n, d, seed=seed)
    if few:   # copies of few rows: equal keys and equal distances
        db = db[np.random.default_rng(seed).integers(0, few, n)]
    q = datagen.make_queries(db, 203, seed=seed + 1)
    if dtype == "f32":
        db, q = datagen.to_f32(db), datagen.to_f32(q)
    return torch.from_numpy(np.ascontiguousarray(db)).cuda(), torch.from_numpy(q).cuda()


@pytest.mark.parametrize("n,d,dtype,curves,m,parts,k,p_max,few", [
    (5000, 128, "u8", 8, 16, 1, 10, 97, 0), (5000, 128, "f32", 8, 16, 1, 10, 64, 0),
    (3001, 64, "u8", 8, 8, 3, 33, 40, 0), (3001, 256, "u8", 16, 16, 8, 1, 5, 0),
    (2000, 64, "f32", 4, 16, 2, 128, 30, 0), (50, 32, "u8", 2, 16, 1, 100, 200, 0),
    (4000, 128, "u8", 8, 16, 1, 10, 300, 9), (40, 16, "u8", 1, 16, 1, 10, 1, 0),
    (2000, 32, "u8", 32, 1, 4, 64, 17, 0), (1000, 128, "u8", 8, 16, 1, 10, 0, 0)])
def test_labels_are_minimal(n, d, dtype, curves, m, parts, k, p_max, few):
    from paper_1209_0410_gb300 import hc
    db, q = rows(n, d, dtype, n + d, few)
    idx = hc.hc_build(db, curves, m, partitions=parts)
    lab = hc.hc_probe_labels(idx, q, k, p_max)
    want, _ = hc.hc_query(idx, q, k, p_max)
    assert int(lab.min()) >= 0 and int(lab.max()) <= p_max
    assert torch.equal(hc.hc_query_depths(idx, q, k, lab)[0], want)
    less, _ = hc.hc_query_depths(idx, q, k, (lab - 1).clamp(min=0))
    assert bool(((less != want).any(1) | (lab == 0)).all())
