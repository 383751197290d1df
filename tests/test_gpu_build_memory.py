"""Device memory that builds take beside the table: the scratch fits the path a
build runs, and a build without enough of it still succeeds."""

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


def _up(x):
    return (x + 255) & ~255


def _placement_bytes(n, m):
    """Arrival counters and an overflow list of a quarter of the keys."""
    return _up(4 * m) + 2 * _up(4 * (n // 4 + 1024))


N, LF = (1 << 24) + 5, 0.95  # 141 MB of slots: beyond the L2, below twice its size


def test_scratch_fits_the_path_of_the_input(G):
    """Page-locked and unaligned arrays are placed ungrouped, pageable ones are inserted as they
    arrive: none of them takes the grouping's scratch."""
    keys, vals = W.make_keys(N + 1, 3), W.make_values(N + 1, 3)
    d_keys, d_vals = keys.cuda(), vals.cuda()
    want = O._u32(vals[:N])
    for arrays, grouped, ranked in (((keys[:N].pin_memory(), vals[:N].pin_memory()), 0, 1),
                                    ((keys[:N].clone(), vals[:N].clone()), 0, 0),
                                    ((d_keys[:N], d_vals[:N]), 1, 1)):
        t = G.HashTable("bcht", N, LF, seed=5)
        t.build(*arrays)
        st = t.stats()
        assert (st["last_build_grouped"], st["last_build_ranked"]) == (grouped, ranked)
        kept = getattr(t, "_scratch_bytes", 0)
        place = _placement_bytes(N, st["num_buckets"])
        assert kept > 4 * place if grouped else kept == ranked * place
        assert (O._u32(t.find(d_keys[:N]).cpu()) == want).all()
    t = G.HashTable("bcht", N, LF, seed=5)
    t.build(d_keys[1:], d_vals[1:])
    assert t.stats()["last_build_ranked"] == 1 and t._scratch_bytes == _placement_bytes(N, t.stats()["num_buckets"])
    assert (O._u32(t.find(d_keys[1:]).cpu()) == O._u32(vals[1:])).all()


@pytest.mark.parametrize("offset", [0, 1])
def test_scratch_of_the_placement_alone_is_used(G, offset):
    """Caller scratch that holds the placement but not the grouping: still a two-phase build."""
    keys, vals = W.make_keys(N + 1, 4).cuda()[offset:N + offset], W.make_values(N + 1, 4).cuda()[offset:N + offset]
    nbytes = G.ght_table_bytes(G.BCHT, N, LF)
    storage = torch.empty(nbytes + 256, dtype=torch.uint8, device="cuda")
    h = G.ght_create_ex(G.BCHT, N, LF, 9, None, _up(storage.data_ptr()), nbytes)
    try:
        need = _placement_bytes(N, G.ght_stats(h).num_buckets)
        assert need < G.ght_build_scratch_bytes(h, N)
        scratch = torch.empty(need + 256, dtype=torch.uint8, device="cuda")
        out = torch.empty_like(vals)
        for given, ranked in ((need, 1), (need - 256, 0)):
            G.ght_set_build_scratch(h, _up(scratch.data_ptr()), given)
            G.ght_build(h, keys, vals, N)
            st = G.ght_stats(h)
            assert (st.last_build_ranked, st.last_build_grouped) == (ranked, 0)
            G.ght_find(h, keys, out, N)
            assert torch.equal(out, vals)
    finally:
        torch.cuda.synchronize()
        G.ght_destroy(h)


def test_a_set_takes_no_scratch_for_values(G):
    """A keys-only build moves keys alone: the grouped arrays hold no values (two levels of about
    4 bytes a key, the placement's counters and list; values would add as much again as the levels)."""
    n = 50_000_000
    t = G.HashTable("bcht_set", n, 0.95, seed=1)
    m = t.stats()["num_buckets"]
    assert G.ght_build_scratch_bytes(t._t, n) < _placement_bytes(n, m) + 2 * 1.1 * 4 * n


def test_a_set_whose_sub_group_outgrows_its_region(G):
    """1300 keys more than average in one 512-bucket sub-group of a set: the attempt is redone with
    exact offsets, which read and write values, in the scratch of a build without them."""
    n, lf, seed = 1 << 22, 0.99, 43
    m = O.num_buckets(n, lf, 32)
    a, c = O.derive_constants(seed, 0, 3)
    cand = np.arange(1, 1 << 24, dtype=np.uint64)
    h0 = ((np.uint64(a[0]) * cand + np.uint64(c[0])) % np.uint64(O.PRIME)) % np.uint64(m)
    crowd = cand[h0 < 512][:1300].astype(np.uint32)
    rest = W.make_keys(n + 4096, 102).numpy().view(np.uint32)
    rest = rest[~np.isin(rest, crowd)][: n - crowd.size]
    keys = torch.from_numpy(np.concatenate([rest, crowd]).view(np.int32).copy())
    t = G.HashTable("bcht_set", n, lf, seed=seed, group_build=1)
    for values in (None, W.make_values(n, 3).cuda()):  # a set ignores values
        t.build(keys.cuda(), values)
        st = t.stats()
        assert (st["attempts"], st["last_build_grouped"], st["last_build_split"]) == (1, 1, 0)
        q = W.make_queries(keys, 1 << 20, 0.5, seed=9)
        want = O.lookup(keys, keys, q) != O.EMPTY
        assert (O._u32(t.find(q.cuda()).cpu()) == want.astype(np.uint32)).all()
    T = O.Table(O.BCHT, n, lf, b=32, m=m)
    T.set_constants(st["hash_a"], st["hash_c"])
    raw = t.export()
    zeros = torch.zeros(n, dtype=torch.int32)
    ok, msg = T.validate(keys, zeros, slots=np.where(raw == O.EMPTY, np.uint64(O.EMPTY_PAIR), raw.astype(np.uint64)))
    assert ok, msg
