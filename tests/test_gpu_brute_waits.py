"""The exact search when waits of its tensor-core kernel run out: a build that looks
at a barrier or a row lock never (every block gives up) or once (some blocks and some
merges do) still gives the oracle's answer, since rows that a block gave up are marked
and searched again."""
import os

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", params=[0, 1])
def impatient(request, tmp_path_factory):
    from paper_1209_0410_gb300 import _build, hc
    _build.build_hc()
    out = tmp_path_factory.mktemp("tries%d" % request.param)
    nvcc, obj, lib = _build._nvcc(), str(out / "brute_tensor.o"), str(out / "libhc_tries.so")
    _build._run([nvcc] + _build.ARCH + _build.NVCC_FLAGS +
                ["-DHC_BRUTE_TRIES=%du" % request.param, "-c",
                 os.path.join(_build.CSRC, "brute_tensor.cu"), "-o", obj])
    others = [os.path.join(_build.BUILD_DIR, f) for f in sorted(os.listdir(_build.BUILD_DIR))
              if f.endswith(".o") and f != "brute_tensor.o"]
    _build._run([nvcc] + _build.ARCH + ["-shared", "-o", lib, obj] + others)
    with hc.use_library(hc.load_library(lib)):
        yield hc


# 313 row tiles are shared by several clusters, which merge in the output rows under a
# lock; fewer than 256 stay with one cluster, whose blocks meet in shared memory
@pytest.mark.parametrize("n,nq,k", [(40_001, 300, 10), (40_001, 90, 16), (34_000, 300, 40),
                                    (20_000, 257, 10), (5000, 1, 1)])
def test_rows_given_up_are_searched_again(impatient, n, nq, k):
    from oracle import oracle as O
    from paper_1209_0410_gb300 import datagen
    db = datagen.make_db(n, 128, seed=n)
    q = datagen.make_queries(db, nq, seed=nq)
    ids, dist = impatient.hc_bruteforce(torch.from_numpy(db).cuda(), torch.from_numpy(q).cuda(), k)
    rids, rdist = O.bruteforce(db, q, k)
    assert np.array_equal(ids.cpu().numpy(), rids)
    assert np.array_equal(dist.cpu().numpy(), O.int32_dist(rdist))
