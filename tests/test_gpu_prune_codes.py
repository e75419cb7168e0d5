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
