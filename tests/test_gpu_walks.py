"""The walks a batch may take -- a warp per query, several warps per query (small
batches), a database in sweeps of ascending ids or partition by partition (large
databases, key order) -- give the same ids and the same distance bits: every row's
distance is summed in one order whoever reads it.  (The warp-per-query walk and the
small batches are checked against the oracle in test_gpu_parity.py and
test_gpu_scale.py.)"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def make(n, d, dtype, nq, seed, few=0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    centres = torch.randint(0, 256, (16, d), generator=g, device="cuda").float()
    db = torch.empty((n, d), dtype=torch.uint8, device="cuda")
    for a in range(0, n, 1 << 20):
        b = min(n, a + (1 << 20))
        which = torch.randint(0, 16, (b - a,), generator=g, device="cuda")
        x = centres[which] + 20 * torch.randn((b - a, d), generator=g, device="cuda")
        db[a:b] = x.round_().clamp_(0, 255).to(torch.uint8)
    if few:
        db = db[torch.randint(0, few, (n,), generator=g, device="cuda")].contiguous()
    q = db[torch.randint(0, n, (nq,), generator=g, device="cuda")].float()
    q = (q + 8 * torch.randn(q.shape, generator=g, device="cuda")).round_().clamp_(0, 255)
    if dtype == "f32":
        return db.float().div_(255.0), q.div_(255.0)
    return db, q.to(torch.uint8)


def same(a, b):
    return torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])


@pytest.mark.parametrize("n,d,dtype,curves,m,parts,k,p,few", [
    (20_000, 128, "u8", 8, 16, 1, 10, 64, 0), (20_000, 64, "u8", 4, 16, 1, 17, 33, 0),
    (9000, 16, "u8", 1, 16, 1, 1, 100, 0), (9000, 48, "u8", 3, 16, 3, 33, 5, 0),
    (9000, 112, "u8", 14, 8, 8, 64, 2, 0), (9000, 256, "u8", 16, 16, 1, 128, 20, 0),
    (9000, 144, "u8", 9, 16, 2, 10, 31, 0), (9000, 16, "f32", 1, 16, 1, 10, 40, 0),
    (9000, 32, "f32", 2, 16, 4, 40, 9, 0), (9000, 128, "f32", 8, 16, 1, 100, 30, 0),
    (9000, 256, "f32", 16, 16, 1, 10, 16, 0), (9000, 48, "f32", 3, 16, 1, 10, 200, 0),
    (3000, 128, "u8", 8, 16, 1, 16, 500, 11), (20, 32, "u8", 2, 16, 1, 30, 64, 0),
    (4000, 64, "u8", 32, 2, 8, 10, 3, 0)])
def test_small_batches_equal_large(n, d, dtype, curves, m, parts, k, p, few):
    from paper_1209_0410_gb300 import hc
    db, q = make(n, d, dtype, 2600, n + d, few)
    idx = hc.hc_build(db, curves, m, partitions=parts)
    want = hc.hc_query(idx, q, k, p)
    depths = torch.from_numpy(np.random.default_rng(n).integers(0, 2 * p, 2600).astype(np.int32))
    depths = depths.cuda()
    deep = hc.hc_query_depths(idx, q, k, depths)
    at = 0
    for b in (1, 2, 7, 39, 152, 153, 305, 1217):
        s = slice(at, at + b)
        qs = q[s].contiguous()
        assert same(hc.hc_query(idx, qs, k, p), [t[s] for t in want]), b
        assert same(hc.hc_query_depths(idx, qs, k, depths[s].contiguous()), [t[s] for t in deep]), b
        pos = hc.hc_query_positions(idx, qs)
        assert same(hc.hc_query_at(idx, qs, k, p, pos), [t[s] for t in want]), b
        at += b
    assert same(hc.hc_query_ordered(idx, q, k, p), want)


@pytest.mark.parametrize("d,curves,m,parts,k,p,nq", [
    (128, 8, 16, 1, 10, 64, 203), (128, 8, 16, 1, 10, 65, 8), (128, 8, 16, 1, 33, 192, 3000),
    (128, 8, 16, 1, 128, 7, 65), (128, 3, 16, 1, 1, 1, 7), (64, 4, 16, 1, 10, 128, 203),
    (64, 4, 8, 1, 10, 129, 203), (16, 1, 16, 1, 10, 512, 99), (48, 3, 16, 1, 40, 171, 99),
    (112, 7, 16, 1, 10, 300, 99), (128, 8, 16, 2, 10, 40, 203), (64, 4, 16, 2, 100, 17, 203),
    (128, 8, 16, 12, 10, 9, 203), (128, 8, 16, 13, 10, 9, 203)])
def test_large_databases_in_key_order(d, curves, m, parts, k, p, nq):
    """350 MB of rows, above the reach of an SM's address translation, few queries."""
    from paper_1209_0410_gb300 import hc
    db, q = make((350 << 20) // d + 13, d, "u8", nq, d + p)
    idx = hc.hc_build(db, curves, m, partitions=parts)
    assert same(hc.hc_query_ordered(idx, q, k, p), hc.hc_query(idx, q, k, p))
    assert same(hc.hc_query_ordered(idx, q, k, 0), hc.hc_query(idx, q, k, 0))


@pytest.mark.parametrize("mb,d,curves,m,parts,k,p,over", [
    (350, 128, 8, 16, 1, 10, 64, 0), (350, 128, 8, 16, 1, 32, 67, 5),
    (350, 128, 3, 16, 1, 1, 171, 1), (350, 128, 8, 16, 1, 33, 200, 3),
    (350, 64, 4, 8, 1, 64, 401, 0), (350, 16, 1, 16, 1, 10, 512, 7),
    (530, 112, 7, 16, 1, 10, 74, 9), (530, 48, 3, 16, 2, 17, 90, 1),
    (450, 128, 8, 16, 2, 10, 32, 2), (350, 128, 8, 16, 2, 10, 64, 4),
    (350, 64, 4, 16, 8, 40, 64, 1), (350, 128, 8, 16, 12, 10, 11, 6),
    (350, 128, 8, 16, 2, 10, 16, 1), (350, 128, 8, 16, 1, 100, 70, 1)])
def test_large_batches_of_large_databases(mb, d, curves, m, parts, k, p, over):
    """Batches that fill the SMs several times: sweeps in key order, whole and cut
    ones, and the walk partition by partition in both orders, at and past the lines
    where they start, equal small batches."""
    from paper_1209_0410_gb300 import hc
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    nq = 4 * sms * 16 + over
    db, q = make((mb << 20) // d + 13, d, "u8", nq, d + p)
    idx = hc.hc_build(db, curves, m, partitions=parts)
    small = [hc.hc_query(idx, q[a:a + 2500].contiguous(), k, p) for a in range(0, nq, 2500)]
    want = [torch.cat([s[i] for s in small]) for i in (0, 1)]
    assert same(hc.hc_query(idx, q, k, p), want)
    assert same(hc.hc_query_ordered(idx, q, k, p), want)
