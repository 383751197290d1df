"""Served pool: what a build takes beside its table comes out of the budget, and
answers written over queries."""

import pytest
import torch

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_07232_gb300 import build
    build.build()
    import paper_2108_07232_gb300 as G
    return G


def test_pool_build_scratch_comes_out_of_the_budget(G):
    """Budgets with room for the table alone, for the placement's scratch too, and for the
    grouping's: the build succeeds, the device memory it takes stays within the budget, and
    used_bytes counts the scratch until the build is done."""
    n, lf = 1 << 25, 0.95  # 283 MB of slots; 76 MB of scratch for the placement, 646 MB with the grouping
    keys, vals = W.make_keys(n, 3).cuda(), W.make_values(n, 3).cuda()
    q = W.make_queries(keys.cpu(), 50001, 0.5, seed=3)
    want = O.lookup(keys.cpu(), vals.cpu(), q)
    table = G.ght_table_bytes(G.BCHT, n, lf)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    for extra, takes in ((1 << 20, False), (80 << 20, False), (700 << 20, True)):
        pool = G.Pool(table + extra)
        most, peak = table + extra, 0
        ticket, tid = pool.submit_build(n, lf, 5, keys, vals)
        while True:
            st = pool.stats()
            peak = max(peak, st["used_bytes"])
            if st["builds_done"]:
                break
        assert pool.wait(ticket)["status"] == 0
        assert peak <= most and pool.stats()["used_bytes"] == table
        if takes:
            assert peak > table
        assert before - torch.cuda.mem_get_info()[0] <= most + (64 << 20)
        d = q.cuda()
        out = torch.empty_like(d)
        torch.cuda.synchronize()
        pool.wait(pool.submit_find(tid, d, out))
        assert (O._u32(out.cpu()) == want).all()
        pool.close()
