"""Launches of one kernel with different shared-memory needs do not get in each
other's way: a kernel's limit on dynamic shared memory belongs to the process, so a
launch that lowered it to its own need could make another thread's launch, or a plan
made earlier, fail."""
import threading

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def make(n, d, seed, queries):
    from paper_1209_0410_gb300 import datagen
    db = datagen.make_db(n, d, seed=seed)
    return torch.from_numpy(db).cuda(), torch.from_numpy(
        datagen.make_queries(db, queries, seed=seed + 1)).cuda()


def race(calls, rounds):
    """Each (function, expected) of calls in its own thread and stream, `rounds` times."""
    errors = []
    start = threading.Barrier(len(calls))

    def work(fn, want):
        stream = torch.cuda.Stream()
        start.wait()
        try:
            with torch.cuda.stream(stream):
                for _ in range(rounds):
                    got = fn(stream)
            stream.synchronize()
            if not all(torch.equal(a, b) for a, b in zip(got, want)):
                errors.append("results differ")
        except Exception as e:   # a refused launch raises here
            errors.append(str(e))

    threads = [threading.Thread(target=work, args=c) for c in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


def query_calls(hc, idx, q, batches, k, p):
    calls = []
    for b in batches:
        qs = q[:b].contiguous()
        ids = torch.empty((b, k), dtype=torch.int32, device="cuda")
        dist = torch.empty((b, k), dtype=torch.int32, device="cuda")
        want = [t.clone() for t in hc.hc_query(idx, qs, k, p)]

        def fn(stream, qs=qs, ids=ids, dist=dist):
            return hc.hc_query(idx, qs, k, p, ids, dist, stream=stream)

        calls.append((fn, want))
    torch.cuda.synchronize()
    return calls


@pytest.mark.parametrize("d,parts", [(128, 1), (128, 16), (256, 4)])
def test_threads_query_one_index_with_batches_of_different_sizes(d, parts):
    from paper_1209_0410_gb300 import hc
    db, q = make(3000, d, 5, 700)
    idx = hc.hc_build(db, 8, 16, partitions=parts)
    race(query_calls(hc, idx, q, (1, 500, 20, 130), 10, 2), 4000)


def test_threads_query_indexes_of_different_list_counts():
    """Batches of one warp per query on indexes of 8 and 128 lists."""
    from paper_1209_0410_gb300 import hc
    db, q = make(3000, 128, 6, 2600)
    calls = []
    for parts in (1, 16):
        idx = hc.hc_build(db, 8, 16, partitions=parts)
        calls += query_calls(hc, idx, q, (2600,), 10, 1)
    race(calls + calls, 3000)


def test_a_plan_without_a_graph_runs_after_a_smaller_plan_was_made():
    from paper_1209_0410_gb300 import hc
    db, q = make(4000, 128, 7, 50)
    config = dict(warps_per_block=16, blocks_per_sm=1, tile=2, use_graph=False)
    many = hc.hc_build(db, 8, 16, partitions=32)
    few = hc.hc_build(db, 8, 16)
    want = hc.hc_query(many, q, 10, 5)
    job = hc.MultiJob(many, q, 10, 5)
    plan = hc.MultiPlan([job], config)
    small = hc.MultiPlan([hc.MultiJob(few, q, 10, 5)], dict(config, warps_per_block=1))
    small.run()
    plan.run()
    torch.cuda.synchronize()
    assert torch.equal(job.ids, want[0]) and torch.equal(job.dist, want[1])
    hc.hc_query_multi([hc.MultiJob(few, q, 10, 5)])
    job.ids.zero_()
    plan.run()
    torch.cuda.synchronize()
    assert torch.equal(job.ids, want[0]) and torch.equal(job.dist, want[1])


def test_threads_run_models_of_different_sizes():
    import numpy as np
    from paper_1209_0410_gb300 import hc
    calls = []
    for dims in ((4, 8, 8), (64, 64, 64)):
        mlp = hc.hc_mlp_create(*dims)
        rng = np.random.default_rng(dims[0])
        mlp.set_params(rng.normal(0, 0.1, mlp.nparam), np.zeros(dims[0]), np.ones(dims[0]))
        x = torch.from_numpy(rng.normal(0, 1, (40, dims[0])).astype(np.float32)).cuda()
        want = [mlp.forward(x, bf16=True)]
        calls.append((lambda s, mlp=mlp, x=x: [mlp.forward(x, bf16=True, stream=s)], want))
    torch.cuda.synchronize()
    race(calls + calls, 3000)
