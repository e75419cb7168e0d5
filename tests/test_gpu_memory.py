"""The device memory that the library keeps between calls: the coded rows' buffer
beside the workspace."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rn():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_17099_gb300 import build as b
    b.build()
    from paper_2602_17099_gb300 import rnsm
    return rnsm


def _coded_search(rn, x, adj, nq):
    # 16 * nq * 256 expected distances: coded rows if that is 8 a row
    q = x[:nq]
    seeds = torch.zeros((nq, 1), dtype=torch.int32, device="cuda")
    return rn.search(x, adj, q, seeds, 256, 5)[0]


def test_a_growing_index_does_not_reallocate_the_codes_each_call(rn):
    # twelve calls, each with 3 % more rows (2.3 MB of codes and more, above the
    # allocator's granularity of 2 MiB): growth by an eighth is four steps at most
    rn.release_workspace()                 # (earlier calls may have left a larger buffer)
    top, d = 430_000, 256
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    x = torch.randn(top, d, generator=g, device="cuda")
    adj = torch.randint(0, 300_000, (top, 2), generator=g, device="cuda", dtype=torch.int32)
    _coded_search(rn, x[:300_000], adj[:300_000], 1300)
    torch.cuda.synchronize()
    free, changes = torch.cuda.mem_get_info()[0], 0
    for i in range(1, 13):
        n = int(300_000 * 1.03 ** i)
        _coded_search(rn, x[:n], adj[:n], 1300)
        now = torch.cuda.mem_get_info()[0]
        changes += now != free
        free = now
    assert 1 <= changes <= 4


def test_kept_codes_give_way_to_the_workspace(rn):
    # a search leaves 1 GB of codes behind; then the caller takes all memory but 256 MB,
    # and a call needs a workspace of some 0.9 GB
    n, d, m, kp = 4_000_000, 256, 20_000_000, 5
    rn.release_workspace()
    x = torch.zeros(n, d, device="cuda")
    x[:, 0] = torch.arange(n, device="cuda") % 1000
    adj = torch.randint(0, n, (n, 1), device="cuda", dtype=torch.int32)
    nplus = torch.randint(0, m, (m, kp), device="cuda", dtype=torch.int32)
    before = torch.cuda.mem_get_info()[0]
    _coded_search(rn, x, adj, 8000)
    assert before - torch.cuda.mem_get_info()[0] > n * d
    outs = torch.empty(m * 14, dtype=torch.int32, device="cuda")   # room for the outputs
    del outs
    hog = torch.empty(torch.cuda.mem_get_info()[0] - (256 << 20), dtype=torch.uint8, device="cuda")
    try:
        offs, ids = rn.reverse_knn(nplus, kp)
        assert int(offs[-1]) == m * kp and ids.shape[0] == m * kp
    finally:
        del hog
        torch.cuda.empty_cache()
        rn.release_workspace()
