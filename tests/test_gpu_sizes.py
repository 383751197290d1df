"""Builds and finds at the sizes where the kernels' splits of the work change:
around a warp's chunk, around one share per warp, and past it."""

import numpy as np
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


def _check(G, scheme, n, lf, seed, n_queries=None, **cfg):
    """Every answer of a fresh build equals the definitional lookup; the layout is valid."""
    keys, vals = W.make_keys(n, seed), W.make_values(n, seed)
    t = G.HashTable(scheme, n, lf, seed=seed, **cfg)
    t.build(keys.cuda(), None if scheme == "bcht_set" else vals.cuda())
    q = W.make_queries(keys, n_queries or n + 9, 0.5, seed=seed + 1)
    got = O._u32(t.find(q.cuda()).cpu())
    want = O.lookup(keys, vals, q)
    if scheme == "bcht_set":
        want = (want != O.EMPTY).astype(want.dtype)
    assert (got == want).all()
    st = t.stats()
    if scheme != "bcht_set":
        T = O.Table(G.SCHEMES[scheme], n, lf, b=st["bucket_size"], m=st["num_buckets"])
        T.set_constants(st["hash_a"], st["hash_c"])
        ok, msg = T.validate(keys, vals, slots=t.export())
        assert ok, msg
    return st


# 3,735,552 pairs: 32 chunks of 32 pairs for each of 152 x 3 x 8 warps
@pytest.mark.parametrize("scheme,lf,n", [("bcht", 0.9, 31), ("bcht", 0.9, 33), ("p2bht", 0.7, 4097),
                                         ("bcht", 0.95, 116736), ("bcht", 0.95, 116737), ("bcht", 0.99, 3735551),
                                         ("iht", 0.8, 3735553), ("p2bht", 0.75, 5000011),
                                         ("iht", 0.8, (1 << 24) + 3)])
def test_insert_shares(G, scheme, lf, n):
    _check(G, scheme, n, lf, seed=n & 0xFFFF)


# around a chunk of 32 queries, a block's 256, and past one chunk per resident warp (4864 x 32)
@pytest.mark.parametrize("nq", [1, 31, 32, 33, 257, 155648, 155649, 700001])
@pytest.mark.parametrize("scheme,b,lf", [("bcht", 16, 0.99), ("p2bht", 16, 0.8), ("iht", 16, 0.8),
                                         ("bcht_lb", 16, 0.9), ("bcht_set", 32, 0.99)])
def test_line_find(G, scheme, b, lf, nq):
    """The default find: answers, sentinel queries and exact probe counts."""
    n = 20011
    keys, vals = W.make_keys(n, 7), W.make_values(n, 7)
    t = G.HashTable(scheme, n, lf, seed=11, count_probes=1, bucket_size=b)
    t.build(keys.cuda(), None if scheme == "bcht_set" else vals.cuda())
    q = W.make_queries(keys, nq, 0.5, seed=nq)
    q[nq // 2::97] = -1
    t.reset_counters()
    got = O._u32(t.find(q.cuda()).cpu())
    want = O.lookup(keys, vals, q)
    if scheme == "bcht_set":
        want = (want != O.EMPTY).astype(want.dtype)
    assert (got == want).all()
    st = t.stats()
    assert st["find_queries"] == nq
    if scheme != "bcht_set":
        T = O.Table(G.SCHEMES[scheme], n, lf, b=b, m=st["num_buckets"])
        T.set_constants(st["hash_a"], st["hash_c"])
        assert st["find_probes"] == T.find(q, slots=t.export())[2]


@pytest.mark.parametrize("tables,most", [(1, 5), (3, 70), (700, 9), (300, 3000)])
def test_batch_line_find_over_uneven_segments(G, tables, most):
    """Tables without keys or queries between others, query segments shorter than a chunk and
    across many of them, sentinel queries: every segment answered from its own table."""
    r = np.random.default_rng(tables)
    nk, nq = r.integers(0, most, tables), r.integers(0, 2 * most, tables) * r.integers(0, 2, tables)
    nq[-1] = 0 if tables > 1 else 7
    ko, qo = (np.concatenate([[0], np.cumsum(x)]).astype(np.uint64) for x in (nk, nq))
    keys, vals = W.make_keys(int(ko[-1]) + 1, 5), W.make_values(int(ko[-1]) + 1, 5)
    q = torch.cat([W.make_queries(keys, int(qo[-1]), 0.8, seed=3), keys[:0]])
    q[3::41] = -1
    b = G.Batch(np.maximum(nk, 1), np.full(tables, 0.9), seed=2)
    b.set_layout(ko, qo)
    got = O._u32(b.run(keys.cuda(), vals.cuda(), q.cuda()).cpu())
    for t in range(tables):
        k0, k1, q0, q1 = (int(x) for x in (ko[t], ko[t + 1], qo[t], qo[t + 1]))
        assert (got[q0:q1] == O.lookup(keys[k0:k1], vals[k0:k1], q[q0:q1])).all(), t


@pytest.mark.parametrize("cfg", [{}, {"tile_lanes": 8}])
def test_pool_requests_of_all_sizes(G, cfg):
    """Requests from one query to several chunks against two tables, a request answered in place,
    sentinel queries; through the direct find and through the gathered one."""
    n = 30000
    pool = G.Pool(1 << 28, **cfg)
    sets = [(W.make_keys(n, s), W.make_values(n, s)) for s in (1, 2)]
    ids = []
    for s, (k, v) in enumerate(sets):
        ticket, table = pool.submit_build(n, 0.95, s, k.cuda(), v.cuda())
        assert pool.wait(ticket)["status"] == 0
        ids.append(table)
    qs = [W.make_queries(sets[i & 1][0], nq, 0.6, seed=i) for i, nq in enumerate([1, 31, 32, 33, 5000, 1, 100003, 64])]
    qs[4][::13] = -1
    ins = [q.cuda() for q in qs]
    outs = [ins[i] if i == 6 else torch.empty_like(q) for i, q in enumerate(ins)]
    torch.cuda.synchronize()
    for ticket in [pool.submit_find(ids[i & 1], q, o) for i, (q, o) in enumerate(zip(ins, outs))]:
        assert pool.wait(ticket)["status"] == 0
    for i, (q, o) in enumerate(zip(qs, outs)):
        assert (O._u32(o.cpu()) == O.lookup(*sets[i & 1], q)).all(), i
    pool.close()


# the one-block build: the smallest tables, a thread's second and last key, the
# most that a block holds, and one key more
@pytest.mark.parametrize("n", [1, 15, 1024, 1025, 20011, 27000, 28500, 32769])
@pytest.mark.parametrize("scheme,lf", [("bcht", 0.96), ("p2bht", 0.75), ("iht", 0.78), ("bcht_lb", 0.9),
                                       ("cuckoo1", 0.6), ("bcht_set", 0.96)])
def test_one_block_build(G, scheme, lf, n):
    st = _check(G, scheme, n, lf if n > 100 else 0.4, seed=n)
    assert st["built"] == 1 and st["n_stored"] == n


def test_one_block_build_reports_sentinels_and_full_tables(G):
    for scheme in ("bcht", "p2bht", "iht", "bcht_lb", "cuckoo1"):
        keys, vals = W.make_keys(3000, 4), W.make_values(3000, 4)
        bad = keys.clone()
        bad[1717] = -1
        t = G.HashTable(scheme, 3000, 0.5, seed=1)
        with pytest.raises(G.GhtError) as e:
            t.build(bad.cuda(), vals.cuda())
        assert e.value.status == "GHT_ERR_SENTINEL_KEY"
        t.build(keys.cuda(), vals.cuda())  # the same table then builds
        assert t.stats()["built"] == 1
    t = G.HashTable("p2bht", 20000, 1.0, seed=1, max_attempts=2)
    with pytest.raises(G.GhtError) as e:
        t.build(W.make_keys(20000, 1).cuda(), W.make_values(20000, 1).cuda())
    assert e.value.status == "GHT_ERR_BUILD_FAILED" and t.stats()["built"] == 0


# placement by load: pairs of keys per thread, odd counts; buckets of 16 and 32, evictions at 0.99
@pytest.mark.parametrize("scheme,b,lf,n", [("p2bht", 16, 0.8, 40001), ("p2bht", 32, 0.88, 622593), ("bcht_lb", 16, 0.99, 622592),
                                           ("bcht_lb", 32, 0.99, 70003), ("p2bht", 16, 0.82, 5000011)])
def test_placement_by_load(G, scheme, b, lf, n):
    st = _check(G, scheme, n, lf, seed=n & 0xFFF, bucket_size=b)
    assert st["last_build_ranked"] == 1 and st["last_build_grouped"] == 0


@pytest.mark.parametrize("n,lf", [(1250003, 0.8), (1250003, 0.6), ((1 << 24) + 77, 0.8)])
def test_cuckoo1_two_phase(G, n, lf):
    """Grouped, one block per sub-group of 4096 slots, the overflow from H_1 (the default from the
    L2's size on, on request below it); odd slot counts."""
    st = _check(G, "cuckoo1", n, lf, seed=n & 0xFFF, n_queries=1 << 20, group_build=1, ranked_build=1)
    assert st["last_build_ranked"] == 1 and st["last_build_grouped"] == 1


def test_batch_overflow_beyond_the_list_rebuilds_the_table(G):
    """Every key of one table in one bucket under its first constants: its overflow outgrows the
    batch's list, and the table is rebuilt alone."""
    n, seed = 6000, 29
    m = O.num_buckets(n, 0.5, 16)
    a, c = O.derive_constants(seed, 0, 3)
    cand = np.arange(1, 1 << 24, dtype=np.uint64)
    h0 = ((np.uint64(a[0]) * cand + np.uint64(c[0])) % np.uint64(O.PRIME)) % np.uint64(m)
    crowd = torch.from_numpy(cand[h0 == h0[0]][:n].astype(np.uint32).view(np.int32).copy())
    assert crowd.numel() == n
    other = W.make_keys(500, 3)
    keys, vals = torch.cat([crowd, other]), W.make_values(n + 500, 8)
    b = G.Batch([n, 500], [0.5, 0.9], seed=seed)
    offs = np.array([0, n, n + 500], dtype=np.uint64)
    b.set_layout(offs, offs)
    out = O._u32(b.run(keys.cuda(), vals.cuda(), keys.cuda()).cpu())
    assert (out == O._u32(vals)).all()
