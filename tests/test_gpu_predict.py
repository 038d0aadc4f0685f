"""The depth predictor's forms: several queries per warp and gaps decided by the
keys' high words, at the edges where either could go wrong.

A batch's depths do not depend on how many queries a warp takes: the whole batch
equals the same queries in slices of one query per warp, bit for bit.  Features of
rows that differ in their lowest bits alone (gaps below, at and just above 2^80,
where the low words decide) equal the oracle's, bit for bit.
"""
import numpy as np
import pytest

from helpers import dev
from oracle import oracle as O
from paper_1209_0410_gb300 import datagen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hc():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1209_0410_gb300 import hc as _hc
    _hc.lib()
    return _hc


def _model(hc, curves, h1, h2):
    rng = np.random.default_rng(curves + h1)
    n_in = 4 * curves
    theta = np.concatenate([rng.normal(0, (2 / n_in) ** 0.5, n_in * h1), rng.normal(0, 0.1, h1),
                            rng.normal(0, (2 / h1) ** 0.5, h1 * h2), rng.normal(0, 0.1, h2),
                            rng.normal(0, 0.5 / h2 ** 0.5, h2), np.full(1, 6.0)])
    mlp = hc.MLP(n_in, h1, h2, 256)
    mlp.set_params(theta.astype(np.float32), np.tile(np.float32([100, 100, 14, 14.5]), curves),
                   1 / np.tile(np.float32([8, 8, 1, 0.5]), curves))
    return mlp


# per SM 32 warps: one query per warp below `resident` queries, two from there (up
# to 8 curves; from 6 x resident with more), four from 2 x resident
@pytest.mark.parametrize("curves,m,d,h1,h2,factor,extra", [
    (8, 16, 128, 64, 64, 1, 0), (8, 16, 128, 64, 64, 2, 3), (8, 16, 128, 33, 20, 2, 1),
    (5, 12, 64, 64, 31, 2, 2), (1, 16, 16, 8, 64, 3, 1), (3, 8, 32, 64, 64, 1, 1),
    (16, 16, 256, 64, 64, 6, 1), (9, 8, 80, 40, 64, 7, 0)])
def test_queries_per_warp(hc, curves, m, d, h1, h2, factor, extra):
    import torch
    resident = torch.cuda.get_device_properties(0).multi_processor_count * 32
    db = datagen.make_db(9001, d, seed=3)
    nq = factor * resident + extra
    q = dev(np.ascontiguousarray(datagen.make_queries(db, 4096, seed=4)[
        np.random.default_rng(5).integers(0, 4096, nq)]))
    idx = hc.hc_build(dev(db), curves, m)
    mlp = _model(hc, curves, h1, h2)
    whole = mlp.predict_depths(idx, q, 0.25, 1, 512)
    parts = torch.cat([mlp.predict_depths(idx, q[a:a + 1000].contiguous(), 0.25, 1, 512)
                       for a in range(0, nq, 1000)])
    assert torch.equal(whole, parts)
    assert whole.min() >= 1 and whole.unique().numel() > 3


@pytest.mark.parametrize("levels", [1, 2, 4, 8, 16, 32])
def test_gaps_of_close_rows(hc, levels):
    """Coordinates that differ in their lowest bits only: the keys share most of
    their high word and the gaps lie on both sides of 2^80."""
    rng = np.random.default_rng(levels)
    db = (np.uint8(96) + rng.integers(0, levels, (3000, 32))).astype(np.uint8)
    q = (np.uint8(96) + rng.integers(0, levels + 1, (200, 32))).astype(np.uint8)
    idx = hc.hc_build(dev(db), 2, 16)
    f = hc.hc_features(idx, dev(q)).cpu().numpy()
    assert np.array_equal(f, O.features(O.build(db, curves=2, m=16), db, q))
