"""CPU check of the bound behind the coded searches (csrc/codes.cu,
code_limit in csrc/search_impl.cuh): with the grid, the residuals and the limit
computed as the kernels do, no row whose code distance exceeds the limit for a
worst entry w has an FP32 distance of w or less."""
import numpy as np
import pytest

F = np.float32


def fp32_dist(q, X, metric):
    acc = np.zeros(len(X), F)
    for j in range(X.shape[1]):            # one chain: the longest accumulation
        t = X[:, j] if metric else q[j] - X[:, j]
        acc = (acc.astype(np.float64) + (q[j].astype(np.float64) * t if metric else t.astype(np.float64) ** 2)).astype(F)
    return F(1) - acc if metric else acc


def codes_of(X):
    lo, hi = X.min(), X.max()
    rng = hi - lo
    s = F(rng / F(255))
    y = X - lo
    c = np.clip(np.rint(y * (F(1) / s)), 0, 255).astype(F)
    r = (y.astype(np.float64) - s.astype(np.float64) * c).astype(F)
    e2 = (r.astype(np.float64) ** 2).sum(1).astype(F).max()
    e = F(1.001) * np.sqrt(e2) + F(1.2e-7) * F(np.sqrt(F(X.shape[1]))) * rng
    norm2 = F(1.0001) * (X.astype(np.float64) ** 2).sum(1).astype(F).max()
    return c.astype(np.int64), s, F(2) * e, norm2


def limit(w, s, err, norm2, metric):
    d2 = w * F(1.0001) if not metric else F(2) * (w + F(1e-4) * norm2 + F(1e-6)) - F(2) + F(2) * norm2
    t = (np.sqrt(np.maximum(d2, F(0))) + err) * (F(1) / s)
    return t * t * F(1.0001) + F(1)


@pytest.mark.parametrize("metric", [0, 1])
@pytest.mark.parametrize("d", [64, 96, 768])
@pytest.mark.parametrize("kind", ["normal", "unit", "offset", "tiny spread", "outlier"])
def test_limit_never_rejects_a_row_that_could_enter(metric, d, kind):
    g = np.random.default_rng(d + metric)
    X = g.standard_normal((400, d))
    X[200:] = X[:200] + 0.2 * X[200:]
    if kind == "unit":
        X /= np.linalg.norm(X, axis=1, keepdims=True)
    elif kind == "offset":
        X = 0.1 * X + 1000.0
    elif kind == "tiny spread":
        X = 1e-3 * X + 1.0
    elif kind == "outlier":
        X[3, 5] = 1e3
    X = X.astype(F)
    c, s, err, norm2 = codes_of(X)
    settled = 0
    for i in range(0, 40):
        dist = fp32_dist(X[i], X, metric)
        S = ((c - c[i]) ** 2).sum(1).astype(F)
        for w in np.quantile(dist, [0.0, 0.01, 0.2, 0.6]).astype(F):
            out = S > limit(F(w), s, err, norm2, metric)
            assert not (out & (dist <= w)).any()
            settled += out.sum()
    if kind == "unit":
        assert settled > 0                 # the bound does settle something
