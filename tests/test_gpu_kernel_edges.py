"""Kernels at the sizes where their tiling can go wrong: edges of tiles and
chunks, remainders, the smallest and largest of each range."""
import numpy as np
import pytest

from oracle import mlp as OM

torch = pytest.importorskip("torch")
E = pytest.importorskip("paper_2504_04018_gb300")

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a), device=DEV)


@pytest.mark.parametrize("B", [1, 7, 8, 9, 2431, 2432, 2433, 5000])
def test_mlp_batch_edges(B):
    """Chunks of 8 rows on at most 304 blocks: part chunks, one chunk per
    block, blocks with one and two chunks. Sums of float32 terms grouped by
    8 rows and then by block: well within 1e-4 of the largest gradient, and
    the same bits when repeated."""
    rng = np.random.default_rng(B)
    F = E.esg_mlp_num_features()
    p = (rng.standard_normal(OM.n_params(F)) * 0.2).astype(np.float32)
    X = (rng.standard_normal((B, F)) * 2 + 0.5).astype(np.float32)
    T = rng.standard_normal((B, 2)).astype(np.float32)
    mu, sigma = rng.standard_normal(F).astype(np.float32), (rng.random(F) + 0.5).astype(np.float32)
    a = (_t(p), _t(X), _t(T), _t(mu), _t(sigma))
    y = E.esg_mlp_forward(a[0], a[1], a[3], a[4]).cpu().numpy()
    ref, _ = OM.forward(p, X, mu, sigma)
    assert np.allclose(y, ref, rtol=1e-5, atol=1e-5)
    loss, g = E.esg_mlp_loss_grad(*a, 0.9)
    again, g2 = E.esg_mlp_loss_grad(*a, 0.9)
    ref_loss, ref_g = OM.loss_and_grad(p, X, T, mu, sigma, 0.9)
    assert abs(loss - ref_loss) <= 1e-5 * max(1.0, abs(ref_loss))
    assert np.max(np.abs(g.cpu().numpy() - ref_g)) <= 1e-4 * np.max(np.abs(ref_g)) + 1e-8
    assert loss == again and torch.equal(g, g2)
