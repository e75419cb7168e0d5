"""The prune over coded rows (csrc/prune_code.cu) against the FP32 kernels:
integer rows (the codes are the rows) and real ones (the codes settle most tests, the
rest is decided in FP32), pools around one and two registers' worth of candidates,
repeats, holes and the owner itself in them, all three row widths, every
reverse-edge pool of a build and a merge, small R and alpha at its extremes."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rn():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_17099_gb300 import build as b
    b.build()
    from paper_2602_17099_gb300 import rnsm
    return rnsm


def _rows(n, d, rng, lo=0):
    c = rng.integers(0, 256, size=(max(2, n // 40), d))
    x = np.clip(c[rng.integers(0, len(c), n)] + rng.integers(-30, 31, size=(n, d)), 0, 255)
    x[0], x[1] = 0, 255
    x[n // 2] = x[n // 3]                      # equal rows: ties by id
    return (x + lo).astype(np.float32)


@pytest.mark.parametrize("d", [64, 96, 128])
@pytest.mark.parametrize("R,L,alpha", [(1, 4, 1.2), (16, 32, 1.2), (32, 64, 1.0), (32, 64, 0.0),
                                       (64, 64, 1.4), (5, 33, 100.0)])
def test_coded_prune_equals_the_oracle(rn, monkeypatch, d, R, L, alpha):
    # the source pools hold R + L / 2 candidates, up to 96: those above 64 take the
    # general kernel
    rng = np.random.default_rng(d + R)
    segs = [_rows(1500, d, rng, -40), _rows(1100, d, rng, -40)]
    graphs = [oracle.build_graph(s, R, L, 1.2) for s in segs]
    want, _ = oracle.rnsm_merge(segs, [g for g, _ in graphs], [e for _, e in graphs],
                                oracle.pair_plan([len(s) for s in segs]), R, L, alpha)
    ts = [(torch.from_numpy(s).cuda(), torch.from_numpy(g).cuda(), e)
          for s, (g, e) in zip(segs, graphs)]
    for (x, g, e) in ts:                       # the build's prunes and reverse edges
        adj, entry = rn.build_segment(x, R, L)
        assert entry == e and torch.equal(adj, g)
    got, st = rn.merge(ts, rn.params(R, L, alpha))
    if R + (L + 1) // 2 <= 64:
        assert st["prune_kernel"][0] == 4
    np.testing.assert_array_equal(got.cpu().numpy(), want)
    for variant in ("0", "3"):
        monkeypatch.setenv("RNSM_PRUNE_VARIANT", variant)
        assert torch.equal(rn.merge(ts, rn.params(R, L, alpha))[0], got)


def _real(kind, n, d, rng):
    x = rng.standard_normal((max(2, n // 40), d))[rng.integers(0, max(2, n // 40), n)]
    x = x + 0.4 * rng.standard_normal((n, d))
    if kind == "unit":
        x /= np.linalg.norm(x, axis=1, keepdims=True)
    elif kind == "close":                      # distances near the codes' step
        x = np.round(x, 1) + 0.01 * rng.standard_normal((n, d))
        x[n // 2:] = x[: n - n // 2] + 1e-3 * rng.standard_normal((n - n // 2, d))
    x[n // 2] = x[n // 3]                      # equal rows: ties by id, distance 0
    return x.astype(np.float32)


@pytest.mark.parametrize("d", [64, 96, 128])
@pytest.mark.parametrize("w", [1, 31, 32, 33, 63, 64])
@pytest.mark.parametrize("kind", ["integers", "unit", "close"])
def test_coded_prune_call_equals_fp32(rn, monkeypatch, kind, d, w):
    rng = np.random.default_rng(w)
    n = 3000
    X = torch.from_numpy(_rows(n, d, rng) if kind == "integers" else _real(kind, n, d, rng)).cuda()
    nv = 2900                                  # enough distances for the rows to be coded
    owners = torch.from_numpy(rng.permutation(n)[:nv].astype(np.int32)).cuda()
    near = (owners.cpu().numpy()[:, None] + 40 * rng.integers(-20, 20, size=(nv, w))) % n
    pool = np.where(rng.random((nv, w)) < 0.1, rng.integers(-1, n, size=(nv, w)), near).astype(np.int32)
    pool[:, 0] = owners.cpu().numpy()          # the owner itself
    if w > 2:
        pool[:, w // 2] = pool[:, 1]           # a repeat
        pool[:, w - 1] = pool[:, 1]            # and another, in the other half
    pool = torch.from_numpy(pool).cuda()
    eu = torch.from_numpy(rng.integers(0, n, 20000).astype(np.int32)).cuda()
    ev = torch.from_numpy(rng.integers(0, n, 20000).astype(np.int32)).cuda()
    lists = torch.from_numpy(rng.integers(-1, n, (n, 24)).astype(np.int32)).cuda()
    res = {}
    for mode in ("0", "1", "2"):
        monkeypatch.setenv("RNSM_SEARCH_CODES", mode)
        res[mode] = [rn.prune(X, owners, pool, 16, a, keep_all_if_fit=k)
                     for a in (0.0, 1.0, 1.2, 50.0) for k in (False, True)]
        res[mode].append(rn.reverse_edges(X, lists.clone(), eu, ev, 1.2))
    for mode in ("1", "2"):
        for a, b in zip(res["0"], res[mode]):
            assert torch.equal(a, b)


@pytest.mark.parametrize("prec", [1, 2])
def test_tile_modes_take_the_coded_walk_on_large_calls(rn, prec):
    rng = np.random.default_rng(3)
    X = torch.from_numpy(_real("unit", 33_500, 96, rng)).cuda()
    segs = [(x, *rn.build_segment(x, 16, 32)) for x in (X[:16_384].clone(), X[16_384:].clone())]
    want, _ = rn.merge(segs, rn.params(16, 32))
    got, st = rn.merge(segs, rn.params(16, 32, prec=prec))
    assert st["prune_kernel"] == [4, 4]
    assert torch.equal(got, want)


def test_a_tuned_choice_of_codes_does_not_outlive_them(rn, monkeypatch):
    # calls large enough to tune, in BF16 mode: with codes (the tuner may choose them),
    # then without, the shape the same
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    X = torch.randn(2000, 64, generator=g, device="cuda")
    X = X[torch.randint(0, 2000, (490_000,), generator=g, device="cuda")]
    X = X + 0.5 * torch.randn(X.shape, generator=g, device="cuda")
    segs = [(x.contiguous(), *rn.build_segment(x.contiguous(), 16, 24)) for x in torch.split(X, 245_000)]
    first, _ = rn.merge(segs, rn.params(16, 24, prec=1))
    monkeypatch.setenv("RNSM_SEARCH_CODES", "0")
    second, st = rn.merge(segs, rn.params(16, 24, prec=1))
    assert 4 not in st["prune_kernel"]
    assert torch.equal(first, second)


def _clusters(n, d, radius, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    c = torch.nn.functional.normalize(torch.randn(n // 200, d, generator=g, device="cuda"), dim=1)
    x = c[torch.randint(0, n // 200, (n,), generator=g, device="cuda")]
    x = x + radius / d ** 0.5 * torch.randn(n, d, generator=g, device="cuda")
    return torch.nn.functional.normalize(x, dim=1).contiguous()


@pytest.mark.parametrize("d", [64, 96, 128])
@pytest.mark.parametrize("radius,coded", [(3.0, True), (0.1, False)])
def test_tight_clusters_are_pruned_over_fp32_rows(rn, monkeypatch, d, radius, coded):
    # neighbours at 0.08 of the distance of rows far apart, the codes' bound at 0.02 of
    # it: most steps of a prune leave a test open, so the codes serve the searches alone
    X = _clusters(20_000, d, radius, d)
    segs = [(x, *rn.build_segment(x, 32, 64)) for x in (X[:10_000].clone(), X[10_000:].clone())]
    got, st = rn.merge(segs, rn.params(32, 64))
    assert (st["prune_kernel"][0] == 4) == coded
    assert (st["prune_kernel"][1] == 4) == coded
    monkeypatch.setenv("RNSM_SEARCH_CODES", "0")
    for x, adj, e in segs:
        a, entry = rn.build_segment(x, 32, 64)
        assert entry == e and torch.equal(a, adj)
    assert torch.equal(rn.merge(segs, rn.params(32, 64))[0], got)


@pytest.mark.parametrize("d", [64, 96, 128])
def test_small_reverse_edge_pools_of_real_rows_take_the_triangle(rn, monkeypatch, d):
    rng = np.random.default_rng(d)
    for kind, n, want in (("wide", 2000, [4, 0]), ("integers", 2000, [4, 4]), ("wide", 8000, [4, 4])):
        X = torch.from_numpy(_rows(2 * n, d, rng)).cuda() if kind == "integers" else _clusters(2 * n, d, 3.0, n)
        segs = [(x, *rn.build_segment(x, 16, 32)) for x in (X[:n].clone(), X[n:].clone())]
        got, st = rn.merge(segs, rn.params(16, 32))
        assert st["prune_kernel"] == want
        monkeypatch.setenv("RNSM_SEARCH_CODES", "0")
        assert torch.equal(rn.merge(segs, rn.params(16, 32))[0], got)
        monkeypatch.delenv("RNSM_SEARCH_CODES")


def _kernels(f):
    """The names of the kernels that a call launches ("" where they cannot be traced)."""
    from torch.profiler import ProfilerActivity, profile
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        f()
        torch.cuda.synchronize()
    return " ".join(e.key for e in prof.key_averages())


# prune calls: distances enough for the rows to be coded (8 a row) from one candidate an
# owner on; reverse edges: on both sides of the list counts from which integers and real
# rows are coded
@pytest.mark.parametrize("d", [64, 96, 128])
@pytest.mark.parametrize("kind", ["integers", "wide"])
def test_coded_calls_run_the_coded_kernel_and_equal_fp32(rn, monkeypatch, kind, d):
    rng = np.random.default_rng(d)
    make = lambda k: torch.from_numpy(_rows(k, d, rng)).cuda() if kind == "integers" else _clusters(k, d, 3.0, k)
    n = 2000
    X = make(n)
    lists = rn.build_segment(X, 32, 64)[0]
    two = torch.cat([lists, lists[lists[:, 0].long().clamp_min(0)]], 1)
    calls = []
    for w, nv in ((1, 8 * n), (2, 8 * n), (33, n), (64, 1536), (64, 1535)):
        owners = torch.from_numpy(rng.integers(0, n, nv)).cuda()
        pool = two[owners, :w].contiguous()
        owners = owners.int()
        calls.append((nv >= 1536, lambda o=owners, p=pool: rn.prune(X, o, p, 16, 1.2)))
    for m in (6143, 6144, 14_335, 14_336):
        Y = make(m)
        adj = rn.build_segment(Y, 32, 64)[0]
        v = torch.arange(m, device="cuda").repeat_interleave(12)
        j = torch.from_numpy(rng.integers(0, 32, (2, len(v)))).cuda()
        u = adj[adj[v, j[0]].long().clamp_min(0), j[1]]
        eu, ev = u[u >= 0].contiguous(), v[u >= 0].int()
        coded = m >= (6144 if kind == "integers" else 14_336)
        calls.append((coded, lambda y=Y, l=adj, a=eu, b=ev: rn.reverse_edges(y, l.clone(), a, b, 1.2)))
    for coded, call in calls:
        monkeypatch.delenv("RNSM_SEARCH_CODES", raising=False)
        got, names = call(), _kernels(call)
        if names:
            assert ("prune_code_kernel" in names) == coded
        monkeypatch.setenv("RNSM_SEARCH_CODES", "0")
        assert torch.equal(call(), got)
