"""The exact search on the tensor cores merges in its output rows and looks at them a
second time: captured in a graph, replayed on other inputs, and run at once on several
streams it gives the oracle's answer."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

# several clusters per query tile (merges under a lock), one cluster, wide rows
SIZES = [(60_000, 128, 300, 10), (9000, 128, 130, 10), (40_000, 256, 100, 40)]


def make(n, d, nq, seed):
    from paper_1209_0410_gb300 import datagen
    db = datagen.make_db(n, d, seed=seed)
    return db, datagen.make_queries(db, nq, seed=seed + 1)


def check(out, db, q, k):
    from oracle import oracle as O
    ids, dist = O.bruteforce(db, q, k)
    assert np.array_equal(out[0].cpu().numpy(), ids)
    assert np.array_equal(out[1].cpu().numpy(), O.int32_dist(dist))


@pytest.mark.parametrize("n,d,nq,k", SIZES)
def test_graph(n, d, nq, k):
    from paper_1209_0410_gb300 import hc
    db, q = make(n, d, nq, 1)
    rows, queries = torch.from_numpy(db).cuda(), torch.from_numpy(q).cuda()
    hc.hc_bruteforce(rows, queries, k)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = hc.hc_bruteforce(rows, queries, k)
    for seed in (1, 5, 9):
        db, q = make(n, d, nq, seed)
        rows.copy_(torch.from_numpy(db))
        queries.copy_(torch.from_numpy(q))
        for t in out:
            t.fill_(7)
        graph.replay()
        torch.cuda.synchronize()
        check(out, db, q, k)


def test_streams():
    from paper_1209_0410_gb300 import hc
    jobs = []
    for i, (n, d, nq, k) in enumerate(SIZES * 2):
        db, q = make(n, d, nq, 20 + i)
        jobs.append((db, q, k, torch.from_numpy(db).cuda(), torch.from_numpy(q).cuda(),
                     torch.cuda.Stream()))
    torch.cuda.synchronize()
    outs = []
    for _ in range(6):
        for db, q, k, rows, queries, stream in jobs:
            with torch.cuda.stream(stream):
                outs.append((hc.hc_bruteforce(rows, queries, k), db, q, k))
    torch.cuda.synchronize()
    first = outs[:len(jobs)]
    for out, db, q, k in first:
        check(out, db, q, k)
    for i, (out, *_) in enumerate(outs):
        want = first[i % len(jobs)][0]
        assert torch.equal(out[0], want[0]) and torch.equal(out[1], want[1])
