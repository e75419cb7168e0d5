"""The visited table of a search (csrc/search_impl.cuh): how many vertices are
evaluated again because it forgot them, and its two forms (ids, and 16-bit tags
for beams over 64) at the graph size where the tags run out of bits."""
import numpy as np
import pytest
import torch

import oracle
from workloads import generators as gen

pytestmark = pytest.mark.gpu

NQ = 1300          # above the latency shape's limit


@pytest.fixture(scope="module")
def rn():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_17099_gb300 import build as b
    b.build()
    from paper_2602_17099_gb300 import rnsm
    return rnsm


@pytest.mark.parametrize("kind,R,most", [("deep", 32, 1.04), ("sift", 32, 1.04), ("embed", 64, 1.12)])
def test_evaluations_stay_near_those_of_an_exact_visited_set(rn, kind, R, most):
    # The oracle's visited set is exact.  A hash of 24 ids a beam entry evaluates up to
    # 1.6 % (R 32) and 9.5 % (R 64: 38 different vertices a beam entry) more, tables of
    # 1,536 or 2,048 ids 15 to 40 % at the larger beams.
    n, metric = 20_000, rn.IP if kind == "embed" else rn.L2
    if kind == "deep":
        X = gen.deep_like(n + NQ, 3)
    elif kind == "embed":
        X = gen.embed_like(n + NQ, 3)
    else:
        segs, Q = gen.sift_case(n_per_seg=n // 2, nq=NQ)
        X = np.concatenate([*segs, Q])
    X, Q = np.ascontiguousarray(X[:n]), np.ascontiguousarray(X[n:])
    x, q = torch.from_numpy(X).cuda(), torch.from_numpy(Q).cuda()
    adj, entry = rn.build_segment(x, R, 2 * R, 1.2, metric)
    seeds = np.full((NQ, 1), entry, np.int32)
    for ef in (64, 128, 256):
        want = oracle.beam_search(X, adj.cpu().numpy(), Q, seeds, ef, 10, metric)[2]
        got = rn.search(x, adj, q, torch.from_numpy(seeds).cuda(), ef, 10, metric, want_ndc=True)[2]
        assert got.double().mean().item() <= most * want.mean(), (ef, got.double().mean(), want.mean())


@pytest.mark.parametrize("n", [300, 1 << 23, (1 << 23) + 1])
def test_searches_on_both_sides_of_the_tags_range(rn, n):
    # ef 128 and lists of 32: 384 buckets, tags of 15 bits for ids below 2^23
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    x = torch.randint(0, 256, (n, 8), generator=g, device="cuda").float()
    adj = torch.randint(-1, n, (n, 32), generator=g, device="cuda", dtype=torch.int32)
    q = torch.randint(0, 256, (NQ, 8), generator=g, device="cuda").float()
    seeds = torch.randint(0, n, (NQ, 2), generator=g, device="cuda", dtype=torch.int32)
    ids, dd, _ = rn.search(x, adj, q, seeds, 128, 20)
    want = oracle.beam_search(x.cpu().numpy(), adj.cpu().numpy(), q.cpu().numpy(), seeds.cpu().numpy(), 128, 20)
    np.testing.assert_array_equal(ids.cpu().numpy(), want[0])
    keep = want[0] >= 0
    np.testing.assert_array_equal(dd.cpu().numpy()[keep], want[1][keep])


def test_the_largest_latency_launch_is_one_wave(rn):
    # 1,216 queries are two CTAs of four on each of 152 SMs: with beams of 256 and their
    # tables both have to fit an SM's shared memory.  In two waves the launch takes twice
    # as long as half of its queries (measured 2.4 times), in one little longer.
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    x = torch.randn(50_000, 8, generator=g, device="cuda")
    adj, entry = rn.build_segment(x, 24, 48)
    q = torch.randn(1216, 8, generator=g, device="cuda")
    seeds = torch.full((1216, 1), entry, dtype=torch.int32, device="cuda")

    def median_ms(nq):
        times = []
        for _ in range(15):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            rn.search(x, adj, q[:nq], seeds[:nq], 256, 10)
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b))
        return sorted(times)[7]

    assert median_ms(1216) < 1.7 * median_ms(608)
