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


def _tables(G, pool, count, n=40000):
    sets, ids = [], []
    for s in range(count):
        k, v = W.make_keys(n, 10 + s), W.make_values(n, 10 + s)
        ticket, tid = pool.submit_build(n, 0.95, s, k.cuda(), v.cuda())
        assert pool.wait(ticket)["status"] == 0
        sets.append((k, v))
        ids.append(tid)
    return sets, ids


@pytest.mark.parametrize("shift", [-4097, -33, -1, 0, 1, 31, 32, 4096])
def test_pool_answers_over_the_queries_of_the_request(G, shift):
    """One request whose answers start `shift` words from its queries, in the same buffer."""
    pool = G.Pool(1 << 28)
    sets, ids = _tables(G, pool, 1)
    n = 300007
    q = W.make_queries(sets[0][0], n, 0.6, seed=8)
    buf = torch.zeros(n + 2 * 5000, dtype=torch.int32, device="cuda")
    ins, out = buf[5000:5000 + n], buf[5000 + shift:5000 + shift + n]
    ins.copy_(q)
    torch.cuda.synchronize()
    assert pool.wait(pool.submit_find(ids[0], ins, out))["status"] == 0
    assert (O._u32(out.cpu()) == O.lookup(*sets[0], q)).all()
    pool.close()


def test_pool_answers_over_the_queries_of_others(G):
    """Requests packed into one launch behind others that keep the pool busy: one is answered over
    the queries of two others, one in place while another asks the same queries."""
    pool = G.Pool(1 << 28)
    sets, ids = _tables(G, pool, 2)
    n = 100003
    qa, qb, qc = (W.make_queries(sets[i & 1][0], n, 0.6, seed=20 + i) for i in range(3))
    a, b, c = (x.cuda() for x in (qa, qb, qc))
    both = torch.cat([a, b])
    out_a, out_b, out_c = (torch.empty_like(a) for _ in range(3))
    busy_q = W.make_queries(sets[0][0], 1 << 22, 0.5, seed=30).cuda()
    busy_out = torch.empty_like(busy_q)
    torch.cuda.synchronize()
    busy = [pool.submit_find(ids[0], busy_q, busy_out) for _ in range(40)]
    half = n // 2
    over = both[half:half + n]  # the end of a's queries and the start of b's
    tickets = [pool.submit_find(ids[0], both[:n], out_a), pool.submit_find(ids[1], both[n:], out_b),
               pool.submit_find(ids[0], c, over), pool.submit_find(ids[1], c, out_c), pool.submit_find(ids[0], c, c)]
    packed = [pool.wait(t)["launch_requests"] for t in tickets]
    for t in busy:
        pool.wait(t)
    assert packed == [len(tickets)] * len(tickets)
    for got, table, q in ((out_a, 0, qa), (out_b, 1, qb), (over, 0, qc), (out_c, 1, qc), (c, 0, qc)):
        assert (O._u32(got.cpu()) == O.lookup(*sets[table], q)).all()
    pool.close()
