"""CPU check of the limits behind the coded prune (limits_of in
csrc/prune_code.cu): with the grid, the residuals and the limits computed as the
kernels do, a test settled by a code distance is settled as the FP32 rule
fmaf(alpha, d(s, c), -d(v, c)) <= 0 settles it."""
import numpy as np
import pytest

from test_code_bound import codes_of, fp32_dist

F = np.float32


def limits(dv, alpha, err, s):
    t = np.sqrt(F(dv) / F(alpha))
    inv = F(1) / s
    a, b = (t * F(0.9998) - err) * inv, (t * F(1.0002) + err) * inv
    return (a * a * F(0.99999) if a > 0 else F(-1)), b * b * F(1.00001) + F(1)


@pytest.mark.parametrize("d", [64, 96, 128])
@pytest.mark.parametrize("kind", ["normal", "unit", "offset", "close"])
def test_limits_settle_as_fp32_does(d, kind):
    g = np.random.default_rng(d)
    X = g.standard_normal((300, d))
    X[100:] = X[g.integers(0, 100, 200)] + 0.3 * X[100:]
    if kind == "unit":
        X /= np.linalg.norm(X, axis=1, keepdims=True)
    elif kind == "offset":
        X = 0.1 * X + 1000.0
    elif kind == "close":
        X[100:] = X[g.integers(0, 100, 200)] + 1e-3 * g.standard_normal((200, d))
    X = X.astype(F)
    c, s, err, _ = codes_of(X)
    D = np.stack([fp32_dist(x, X, 0) for x in X])
    S = np.stack([((c - q) ** 2).sum(1).astype(F) for q in c])
    settled = total = 0
    for alpha in (0.5, 1.0, 1.2, 3.0):
        for v in range(0, 30):
            for w in range(30, 300, 9):
                yes, no = limits(D[v, w], alpha, err, s)
                rule = F(alpha) * D[:, w].astype(np.float64) - np.float64(D[v, w]) <= 0
                assert rule[S[:, w] <= yes].all()
                assert not rule[S[:, w] > no].any()
                settled += (S[:, w] <= yes).sum() + (S[:, w] > no).sum()
                total += len(X)
    if kind in ("normal", "unit"):
        assert settled > 0.9 * total
