"""Small batches, several warps to a query: every number of warps (2, 4, 8 in a block
of eight, 16) gives the ids and distance bits of a warp per query, and small batches on
many streams share the chip."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,dtype,curves,parts,k,p", [
    (30_000, 128, "u8", 8, 1, 10, 64), (30_000, 128, "u8", 8, 1, 100, 600),
    (30_000, 96, "u8", 6, 2, 33, 20), (30_000, 96, "u8", 6, 1, 10, 17),
    (30_000, 64, "u8", 4, 1, 10, 150), (20_000, 256, "u8", 16, 1, 10, 130),
    (20_000, 528, "u8", 8, 2, 100, 40), (20_000, 128, "f32", 8, 1, 10, 130),
    (20_000, 16, "f32", 1, 4, 40, 100), (20_000, 32, "f32", 2, 1, 10, 300)])
def test_every_number_of_warps(n, d, dtype, curves, parts, k, p):
    from paper_1209_0410_gb300 import hc
    g = torch.Generator(device="cuda").manual_seed(n + d)
    db = torch.randint(0, 256, (n, d), generator=g, device="cuda").to(torch.uint8)
    q = torch.randint(0, 256, (3000, d), generator=g, device="cuda").to(torch.uint8)
    if dtype == "f32":
        db, q = db.float().div_(255.0), q.float().div_(255.0)
    idx = hc.hc_build(db, curves, 16, partitions=parts)
    want = hc.hc_query(idx, q, k, p)   # a warp per query
    pos = hc.hc_query_positions(idx, q)
    depths = torch.full((3000,), p, dtype=torch.int32, device="cuda")
    for b in (1, 30, 57, 58, 113, 114, 115, 152, 228, 229, 300, 456, 700, 1215):
        rows = [t[:b] for t in want]
        qs = q[:b].contiguous()
        for got in (hc.hc_query(idx, qs, k, p), hc.hc_query_at(idx, qs, k, p, pos[:b].contiguous()),
                    hc.hc_query_depths(idx, qs, k, depths[:b].contiguous())):
            assert torch.equal(got[0], rows[0]) and torch.equal(got[1], rows[1]), b


def test_small_batches_on_many_streams_share_the_chip():
    """320 batches of 400 queries on 16 streams take little longer than their queries
    in 20 batches of 6,400 one after the other (1.05 times; 2.1 when a batch keeps each
    SM to itself).  Everything is queued before the first one runs."""
    from paper_1209_0410_gb300 import datagen, hc
    db = torch.from_numpy(datagen.make_db(100_000, 128, seed=3)).cuda()
    idx = hc.hc_build(db, 8, 16)
    q = db[torch.randint(0, 100_000, (6400,), device="cuda")].contiguous()
    parts = [q[400 * i:400 * (i + 1)].contiguous() for i in range(16)]
    out = [hc.hc_query(idx, x, 10, 64) for x in parts]
    big = hc.hc_query(idx, q, 10, 64)
    streams = [torch.cuda.Stream() for _ in parts]

    def many(main):
        for s in streams:
            s.wait_stream(main)
        for _ in range(20):
            for s, x, o in zip(streams, parts, out):
                hc.hc_query(idx, x, 10, 64, *o, stream=s)
        for s in streams:
            main.wait_stream(s)

    def one(main):
        for _ in range(20):
            hc.hc_query(idx, q, 10, 64, *big)

    def fastest(fn):
        times = []
        for _ in range(6):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            torch.cuda.synchronize()
            torch.cuda._sleep(80_000_000)   # 40 ms, in which everything is queued
            a.record()
            fn(torch.cuda.current_stream())
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return min(times)

    times = fastest(many), fastest(one)
    assert torch.equal(torch.cat([o[0] for o in out]), big[0])
    assert times[0] < 1.6 * times[1], times
