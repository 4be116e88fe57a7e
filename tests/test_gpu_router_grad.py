"""GPU: the router's gradient kernel at the edges of its tiles (16 and 64 rows;
64-row tiles from 64 x 152 rows on), against the FP64 reference."""
import numpy as np
import pytest

from oracle import router as R
from paper_2507_09772_gb300 import jk

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def blob(seed):
    rng = np.random.default_rng(seed)
    b = jk.JkRouterBlob()
    b.magic, b.version, b.margin, b.quantile = jk.ROUTER_MAGIC, 1, 0.0, 0.9
    th = (0.2 * rng.standard_normal(jk.ROUTER_NPARAM)).astype(np.float32)
    mu = (0.3 * rng.standard_normal(16)).astype(np.float32)
    isd = (0.5 + rng.random(16)).astype(np.float32)
    b.theta[:], b.mu[:], b.isd[:] = th.tolist(), mu.tolist(), isd.tolist()
    return b, th, mu, isd


def rows(n, seed):
    rng = np.random.default_rng(seed)
    return rng.standard_normal((n, 12)).astype(np.float32), rng.standard_normal(n).astype(np.float32)


def rows_with_a_heavy_tail(n, seed):
    """Rows of which those in the last tile (the last n % 64, or 64) carry nearly
    all of the loss and the gradient, each at least a two-hundredth of it: large
    features, along one direction with a different factor each, and labels far off."""
    X, y = rows(n, seed)
    tail = n % 64 or min(n, 64)
    rng = np.random.default_rng(seed + 1)
    X[n - tail:] = (3e4 * (1.0 + 0.2 * rng.random((tail, 1))) * np.ones(12)).astype(np.float32)
    X[n - tail:] += (3e3 * rng.standard_normal((tail, 12))).astype(np.float32)
    y[n - tail:] = 1e9 * (1.0 + rng.random(tail))
    return X, y, tail


@pytest.mark.parametrize("n", [1, 15, 16, 17, 63, 64, 65, 4864, 4865, 9664, 9728, 9729, 30011, 65536])
@pytest.mark.parametrize("noalloc", [False, True])
def test_gradient_at_tile_edges(n, noalloc):
    """A lost or doubled row of the last tile shows: without any one of them the
    reference itself is further off than twice the tolerance."""
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    b, th, mu, isd = blob(n)
    X, y, tail = rows_with_a_heavy_tail(n, n + 1)
    f = jk.jk_router_gradient_noalloc if noalloc else jk.jk_router_gradient
    g, loss = f(b, torch.tensor(X, device="cuda"), torch.tensor(y, device="cuda"), 0.9)
    lref, gref = R.pinball_grad(th, mu, isd, X, y, 0.9)
    # the loss: FP32 products and FP64 sums; the gradient: activations an FP32 rounding away from a
    # BF16 tie (2^-8 of one of 64 inputs: 5e-4 of a row's gradient, a few of them in a single row)
    tol_l, tol_g = 1e-5, 5e-3
    assert loss == pytest.approx(lref, rel=tol_l)
    assert np.linalg.norm(g - gref) <= tol_g * np.linalg.norm(gref)
    for k in (n - tail, n - tail // 2 - 1, n - 1):
        if n > 1:
            l1, g1 = R.pinball_grad(th, mu, isd, np.delete(X, k, 0), np.delete(y, k), 0.9)
            l1, g1 = l1 * (n - 1) / n, g1 * (n - 1) / n
            assert abs(l1 - lref) > 2 * tol_l * lref
            assert np.linalg.norm(g1 - gref) > 2 * tol_g * np.linalg.norm(gref)


def test_infinite_feature_leaves_inactive_units_alone():
    """A row with an infinite feature: units it drives to -inf are inactive and
    take no gradient from it; no NaN appears in their weights."""
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    b, th, mu, isd = blob(5)
    W1 = th[:768].reshape(12, 64)
    X, y = rows(100, 6)
    X[3, 2] = np.inf
    g, _ = jk.jk_router_gradient(b, torch.tensor(X, device="cuda"), torch.tensor(y, device="cuda"), 0.9)
    dead = W1[2] < 0
    dW1 = g[:768].reshape(12, 64)[:, dead]
    assert np.isfinite(dW1).all() and np.isfinite(g[1024:1088][dead]).all()
