"""Searches over coded rows (a byte per dimension; csrc/codes.cu) against the
FP32 searches: RNSM_SEARCH_CODES forces 0 FP32 rows only, 1 codes as a filter,
2 (default) codes alone where they are the rows.  Ids and distances are the
same bit for bit, whatever the data, the metric and the shape of the beam."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

NQ = 1300          # above the latency shape's limit, which takes no codes


@pytest.fixture(scope="module")
def rn():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_17099_gb300 import build as b
    b.build()
    from paper_2602_17099_gb300 import rnsm
    return rnsm


def _rows(kind, n, d, rng):
    if kind == "bytes":                      # exact codes, both ends of the grid
        x = rng.integers(0, 256, size=(n, d))
        x[0], x[1] = 0, 255
    elif kind == "negative integers":        # span 255 around an offset
        x = rng.integers(-1100, -844, size=(n, d))
    elif kind == "wide integers":            # span 256: not codes, a filter
        x = rng.integers(0, 257, size=(n, d))
        x[0], x[1] = 0, 256
    elif kind == "constant":                 # range 0, every distance a tie
        x = np.full((n, d), 3.0)
    else:
        x = rng.standard_normal((n, d))
        x[n // 2:] = x[: n - n // 2] + 0.3 * x[n // 2:]     # near neighbours
        if kind == "unit":
            x /= np.linalg.norm(x, axis=1, keepdims=True)
        elif kind == "offset":               # the spread is a thousandth of the norm
            x = 0.1 * x + 1000.0
        elif kind == "outlier":              # one component stretches the grid
            x[7, 3] = 3e4
    return x.astype(np.float32)


def _graph(n, r, rng):
    adj = rng.integers(-1, n, size=(n, r)).astype(np.int32)     # holes among them
    adj[:, -1] = adj[:, 0]                                       # a repeated neighbour
    return adj


def _search(rn, monkeypatch, mode, X, adj, Q, seeds, ef, k, metric):
    monkeypatch.setenv("RNSM_SEARCH_CODES", str(mode))
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    ids, dd, _ = rn.search(t(X), t(adj), t(Q), t(seeds), ef, k, metric)
    return ids.cpu().numpy(), dd.cpu().numpy()


@pytest.mark.parametrize("d", [64, 96, 128, 256, 768])
@pytest.mark.parametrize("kind", ["bytes", "negative integers", "wide integers", "constant",
                                  "normal", "unit", "offset", "outlier"])
def test_coded_search_equals_fp32_search(rn, monkeypatch, d, kind):
    rng = np.random.default_rng(d)
    X = _rows(kind, 2001, d, rng)
    adj = _graph(len(X), 32, rng)
    Q = X[rng.integers(0, len(X), NQ)].copy()
    seeds = rng.integers(-1, len(X), size=(NQ, 3)).astype(np.int32)
    for metric in (rn.L2, rn.IP):
        for ef, k in ((33, 10), (64, 64)):
            want = _search(rn, monkeypatch, 0, X, adj, Q, seeds, ef, k, metric)
            for mode in (1, 2):
                got = _search(rn, monkeypatch, mode, X, adj, Q, seeds, ef, k, metric)
                np.testing.assert_array_equal(got[0], want[0])
                np.testing.assert_array_equal(got[1], want[1])


@pytest.mark.parametrize("r_in", [1, 31, 33, 64, 70])
@pytest.mark.parametrize("ef,k,n_seeds", [(1, 1, 1), (32, 32, 33), (100, 7, 64), (256, 256, 1)])
def test_coded_search_shapes(rn, monkeypatch, r_in, ef, k, n_seeds):
    # list lengths around one and two batches, beams at their register steps, and
    # queries that are no rows (their own residuals; off the rows' range)
    rng = np.random.default_rng(r_in)
    for kind, stretch in (("unit", 1.02), ("bytes", 1.0)):
        X = _rows(kind, 3000, 96, rng)
        Q = (_rows(kind, NQ, 96, rng) * np.float32(stretch)).astype(np.float32)
        adj = _graph(len(X), r_in, rng)
        seeds = rng.integers(0, len(X), size=(NQ, n_seeds)).astype(np.int32)
        want = _search(rn, monkeypatch, 0, X, adj, Q, seeds, ef, k, rn.L2)
        for mode in (1, 2):
            got = _search(rn, monkeypatch, mode, X, adj, Q, seeds, ef, k, rn.L2)
            np.testing.assert_array_equal(got[0], want[0])
            np.testing.assert_array_equal(got[1], want[1])


@pytest.mark.parametrize("kind", ["bytes", "unit"])
def test_coded_merge_build_and_expand_equal_fp32(rn, monkeypatch, kind):
    rng = np.random.default_rng(5)
    X = torch.from_numpy(_rows(kind, 9000, 96, rng)).cuda()
    parts = [X[:2500].contiguous(), X[2500:6000].contiguous(), X[6000:].contiguous()]
    plan = [(0, 1), (0, 2), (1, 2)]
    out = {}
    for mode in (0, 1, 2):
        monkeypatch.setenv("RNSM_SEARCH_CODES", str(mode))
        graphs = [rn.build_segment(p, 16, 32) for p in parts]
        segs = [(p, g, e) for p, (g, e) in zip(parts, graphs)]
        merged = [rn.merge(segs, rn.params(16, 32, 1.2, flags=f), plan)[0]
                  for f in (0, rn.FLAG_CM, rn.FLAG_GRAPH, rn.FLAG_GRAPH)]
        out[mode] = [g for g, _ in graphs] + [rn.expand(parts[2], graphs[2][0], 16)] + merged
    for mode in (1, 2):
        for a, b in zip(out[mode], out[0]):
            assert torch.equal(a, b)


@pytest.mark.parametrize("d", [64, 96, 128, 256, 768])
@pytest.mark.parametrize("kind,mode", [("bytes", 2), ("unit", 1), ("outlier", 0)])
def test_the_searches_run_in_the_mode_that_the_rows_allow(rn, monkeypatch, d, kind, mode):
    # the kernel's third template argument: 0 FP32 rows, 1 codes first, 2 codes alone (not
    # at 768 dimensions, whose distances can exceed 2^24)
    from torch.profiler import ProfilerActivity, profile
    rng = np.random.default_rng(d)
    X = _rows(kind, 2001, d, rng)
    adj = _graph(len(X), 32, rng)
    Q = X[rng.integers(8, len(X), NQ)].copy()
    seeds = rng.integers(0, len(X), size=(NQ, 1)).astype(np.int32)
    _search(rn, monkeypatch, 2, X, adj, Q, seeds, 64, 10, rn.L2)
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        _search(rn, monkeypatch, 2, X, adj, Q, seeds, 64, 10, rn.L2)
        torch.cuda.synchronize()
    names = [e.key for e in prof.key_averages() if "search_kernel<" in e.key]
    want = 1 if d == 768 and mode == 2 else mode
    for name in names:                         # (none where kernels cannot be traced)
        assert name.split("search_kernel<")[1].split(",")[2].strip() == str(want), name
