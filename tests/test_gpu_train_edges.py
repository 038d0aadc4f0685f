"""Gradients, one Adam step and the FP32 outputs of the training kernels at the
edges of their tiles (32 samples per block, 64 per stage, 4 x 8 weights per warp,
layers padded to 64 units) against the oracle's float64 backpropagation.

Tolerance: a gradient is a float32 sum of n products of values that passed three
layers of at most 64 terms, so its error is below (n + 200) 2^-24 of the largest
sum of absolute terms; 2e-4 of the largest gradient holds for n <= 3,000."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp as OM  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(1, 1, 1), (5, 7, 3), (32, 64, 64), (33, 9, 64), (64, 63, 17)])
@pytest.mark.parametrize("n,max_batch", [(1, 1), (31, 40), (32, 32), (33, 33), (64, 100), (65, 65),
                                         (257, 300), (2977, 3001)])
def test_step_against_float64(dims, n, max_batch):
    from paper_1209_0410_gb300 import hc
    rng = np.random.default_rng(n * 100 + dims[0])
    X = rng.normal(3.0, 2.0, (n, dims[0])).astype(np.float32)
    T = rng.normal(2.0, 1.0, n).astype(np.float32)
    theta = OM.init(5, *dims).astype(np.float32)
    theta += rng.normal(0, 0.05, theta.size).astype(np.float32)
    mu = np.full(dims[0], 3.0, np.float32)
    isd = np.full(dims[0], 0.5, np.float32)
    mlp = hc.MLP(*dims, max_batch=max_batch)
    mlp.set_params(theta, mu, isd)
    x, t = torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda()
    g, loss = mlp.gradients(x, t)
    g = g.cpu().numpy().astype(np.float64)
    th = theta.astype(np.float64)
    ref, ref_loss = OM.gradients(th, mu, isd, X.astype(np.float64), T.astype(np.float64), *dims)
    assert np.max(np.abs(g - ref)) <= 2e-4 * np.abs(ref).max()
    assert loss == pytest.approx(ref_loss, rel=1e-4)
    y, _ = OM.forward(th, mu, isd, X.astype(np.float64), *dims)
    assert np.allclose(mlp.forward(x).cpu().numpy(), y, rtol=1e-5, atol=1e-5)
    mlp.train_step(x, t, 1e-3)
    z = np.zeros(len(theta))
    assert np.max(np.abs(mlp.get_params()[0] - OM.adam_step(th, g, z, z, 1, 1e-3)[0])) <= 1e-6
    mlp.free()


@pytest.mark.parametrize("n,n_in", [(256, 1), (257, 32), (4095, 33), (10_000, 64)])
def test_normalisation_statistics(n, n_in):
    """mu and isd of a training run: float64 sums, so equal to numpy's to the
    last float32 rounding; a constant column has isd 1000."""
    from paper_1209_0410_gb300 import hc
    rng = np.random.default_rng(n)
    X = rng.normal(100.0, 7.0, (n, n_in)).astype(np.float32)
    X[:, n_in // 2] = 42.0
    mlp = hc.MLP(n_in, 4, 4, max_batch=256)
    mlp.set_params(OM.init(1, n_in, 4, 4).astype(np.float32), np.zeros(n_in), np.ones(n_in))
    mlp.fit(torch.from_numpy(X).cuda(), torch.ones(n, dtype=torch.int32).cuda(), 1, 256, 1e-3)
    _, mu, isd = mlp.get_params()
    ref = X.astype(np.float64)
    assert np.allclose(mu, ref.mean(0), rtol=2e-7, atol=0)
    sd = ref.std(0, ddof=1)
    assert np.allclose(isd, 1.0 / np.maximum(sd, 1e-3), rtol=2e-7, atol=0)
    mlp.free()
