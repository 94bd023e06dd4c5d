"""Loss and gradient of the initial-guess model at the edges of its tiles against NumPy in 64 bits."""
import numpy as np
import pytest

from paper_2010_04768_gb300 import gfcc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="session", autouse=True)
def _built():
    from paper_2010_04768_gb300 import build
    build.build()
    gfcc.load()


def reference(w, h, F, G):
    W1, b1, W2, b2, W3, b3, mu, sd = np.split(w, np.cumsum([27 * h, h, h * h, h, 16 * h, 16, 27]))
    W1, W2, W3 = W1.reshape(h, 27), W2.reshape(h, h), W3.reshape(16, h)
    X = (F - mu) / sd
    Z1 = X @ W1.T + b1
    H1 = np.maximum(Z1, 0)
    Z2 = H1 @ W2.T + b2
    H2 = np.maximum(Z2, 0)
    Y = H2 @ W3.T + b3
    c = Y[:, ::2] + 1j * Y[:, 1::2]
    a = np.concatenate([c.sum(1, keepdims=True) - 1, c], axis=1)
    Ga = np.einsum("sjl,sl->sj", G, a)
    g00 = G[:, 0, 0].real
    on = g00 > 0
    inv = np.where(on, 1.0 / np.where(on, g00, 1.0), 0.0)
    loss = np.einsum("sj,sj->s", a.conj(), Ga).real * inv
    d = 2 * (Ga[:, :1] + Ga[:, 1:]) * inv[:, None] / F.shape[0]
    dY = np.stack([d.real, d.imag], axis=2).reshape(-1, 16)
    dZ2 = (dY @ W3) * (Z2 > 0)
    dZ1 = (dZ2 @ W2) * (Z1 > 0)
    parts = [dZ1.T @ X, dZ1.sum(0), dZ2.T @ H1, dZ2.sum(0), dY.T @ H2, dY.sum(0), np.zeros(54)]
    return loss.mean(), np.concatenate([p.ravel() for p in parts])


# one unit and one sample; a ragged tile; a whole number of tiles; sums longer than two steps of K; a batch whose
# staging exceeds the pinned buffer
@pytest.mark.parametrize("hidden,batch", [(1, 1), (31, 17), (100, 130), (256, 300), (64, 12000)])
@pytest.mark.parametrize("precision", [gfcc.MLP_FP32, gfcc.MLP_FP64])
def test_loss_grad_matches_numpy(hidden, batch, precision):
    rng = np.random.default_rng(hidden + batch)
    w = np.concatenate([rng.standard_normal(27 * hidden) / 5, rng.standard_normal(hidden) / 10,
                        rng.standard_normal(hidden ** 2) / np.sqrt(hidden), rng.standard_normal(hidden) / 10,
                        rng.standard_normal(16 * hidden) / np.sqrt(hidden), rng.standard_normal(16) / 10,
                        rng.standard_normal(27) / 10, 1 + rng.random(27)])
    F = rng.standard_normal((batch, 27))
    U = rng.standard_normal((batch, 9, 12)) + 1j * rng.standard_normal((batch, 9, 12))
    G = U.conj() @ U.transpose(0, 2, 1)
    G[batch // 2 if batch > 1 else 1:][:1] = 0   # a sample without a right-hand side
    w32 = w if precision == gfcc.MLP_FP64 else w.astype(np.float32).astype(np.float64)
    m = gfcc.MLP(w, hidden, precision)
    m.set_params(w)
    loss, grad = m.loss_grad(F, G)
    m.close()
    ref_loss, ref = reference(w32, hidden, F, G)
    # sums of at most max(hidden, batch) terms, five layers deep; a ReLU within rounding of zero may switch in FP32,
    # which moves one sample's share of a gradient entry
    u = 2.0 ** -53 if precision == gfcc.MLP_FP64 else 2.0 ** -24
    tol = 20 * u * np.sqrt(max(hidden, batch, 27)) * 5
    assert abs(loss - ref_loss) <= tol * abs(ref_loss)
    assert np.linalg.norm(grad - ref) <= tol * np.linalg.norm(ref)
    assert np.all(grad[-54:] == 0)
