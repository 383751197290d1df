"""Builds on the paths beside the default one, and the lines between the paths."""

import ctypes

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


def _check(G, t, scheme, keys, vals, b=None):
    """Valid layout and definitional answers of a built table; its stats."""
    st = t.stats()
    sets = scheme == "bcht_set"
    q = W.make_queries(keys, min(keys.numel(), 1 << 20) + 9, 0.5, seed=17)
    got = O._u32(t.find(q.cuda()).cpu())
    want = O.lookup(keys, vals, q)
    assert (got == ((want != O.EMPTY).astype(want.dtype) if sets else want)).all()
    T = O.Table(O.BCHT if sets else G.SCHEMES[scheme], keys.numel(), 0.5, b=st["bucket_size"],
                t=st["threshold"] or None, m=st["num_buckets"])
    T.set_constants(st["hash_a"], st["hash_c"])
    slots = t.export()
    if sets:
        slots = np.where(slots == O.EMPTY, np.uint64(O.EMPTY_PAIR), slots.astype(np.uint64))
        vals = torch.zeros_like(vals)
    ok, msg = T.validate(keys, vals, slots=slots)
    assert ok, msg
    return st


@pytest.mark.parametrize("scheme,lf,n,ranked", [("iht", 0.78, 21000, 0), ("iht", 0.78, 22000, 1), ("iht", 0.6, 19000, 1),
                                                ("p2bht", 0.6, 19000, 1), ("bcht", 0.95, 18000, 0),
                                                ("bcht_set", 0.95, 27000, 0)])
def test_one_block_builds_from_page_locked_arrays(G, scheme, lf, n, ranked):
    """Values that do not fit beside the keys and leave no room for L1 are not gathered over the
    host link: such builds run in two phases from page-locked arrays, in one block from others."""
    keys, vals = W.make_keys(n, 5), W.make_values(n, 5)
    for place, two_phase in ((lambda x: x.pin_memory(), ranked), (lambda x: x.cuda(), 0), (lambda x: x, 0)):
        t = G.HashTable(scheme, n, lf, seed=3)
        t.build(place(keys), None if scheme == "bcht_set" else place(vals))
        st = _check(G, t, scheme, keys, vals)
        assert st["last_build_ranked"] == two_phase and (st["last_fill_ms"] == 0.0) == (not two_phase)


def test_bucket_size_one_is_placed_ungrouped_only_on_request(G):
    """Between the L2's size and twice it: arrays off a 16-byte boundary and page-locked ones, which
    build ungrouped, are inserted in input order; the ungrouped placement on request."""
    n, lf = (1 << 24) + 3, 0.8  # 168 MB of slots
    keys, vals = W.make_keys(n + 1, 6), W.make_values(n + 1, 6)
    dk, dv = keys.cuda(), vals.cuda()
    for cfg, k, v, ranked in (({}, dk[1:], dv[1:], 0), ({"ranked_build": 1}, dk[1:], dv[1:], 1),
                              ({}, keys[:n].pin_memory(), vals[:n].pin_memory(), 0)):
        t = G.HashTable("cuckoo1", n, lf, seed=2, **cfg)
        t.build(k, v)
        st = _check(G, t, "cuckoo1", k.cpu(), v.cpu())
        assert (st["last_build_ranked"], st["last_build_grouped"]) == (ranked, 0)


def test_one_block_builds_of_many_sizes_keep_nothing_per_size(G):
    """Builds of 4000 different key counts leave nothing behind on the host heap."""
    class Info(ctypes.Structure):
        _fields_ = [(f, ctypes.c_size_t) for f in ("arena", "ordblks", "smblks", "hblks", "hblkhd", "usmblks",
                                                   "fsmblks", "uordblks", "fordblks", "keepcost")]
    libc = ctypes.CDLL("libc.so.6")
    libc.mallinfo2.restype = Info
    n = 4400
    keys, vals = W.make_keys(n, 7).cuda(), W.make_values(n, 7).cuda()
    t = G.HashTable("bcht", n, 0.9, seed=1)
    for i in range(1, 401):
        t.build(keys[:i], vals[:i])
    before = libc.mallinfo2().uordblks
    for i in range(401, n + 1):
        t.build(keys[:i], vals[:i])
    # 4000 cached sizes of a hash map took over 128 KB
    assert libc.mallinfo2().uordblks - before < 64 << 10


# the most keys a scheme builds in one block, and one more
@pytest.mark.parametrize("scheme,lf,most", [("bcht", 0.96, 18432), ("bcht", 0.97, 8192), ("bcht", 0.99, 8192),
                                            ("cuckoo1", 0.6, 2048), ("p2bht", 0.75, 20480), ("bcht_lb", 0.9, 20480)])
@pytest.mark.parametrize("more", [0, 1])
def test_the_most_keys_of_a_one_block_build(G, scheme, lf, most, more):
    n = most + more
    keys, vals = W.make_keys(n, n & 0xFF), W.make_values(n, 9)
    t = G.HashTable(scheme, n, lf, seed=n)
    t.build(keys.cuda(), vals.cuda())
    st = _check(G, t, scheme, keys, vals)
    assert st["last_build_small"] == 1 - more and st["built"] == 1


# the most that fits 226 KB: keys, one index a slot, one count a bucket
@pytest.mark.parametrize("scheme,lf,b", [("iht", 0.78, 16), ("iht", 0.8, 32), ("bcht_set", 0.95, 32)])
def test_the_largest_one_block_build(G, scheme, lf, b):
    def fits(n):
        return 4 * (n + O.num_buckets(n, lf, b) * (b + 1)) <= 226 * 1024

    most = max(n for n in range(20000, 32769) if fits(n))
    for n in (most, most + 1):
        keys, vals = W.make_keys(n, 4), W.make_values(n, 4)
        t = G.HashTable(scheme, n, lf, seed=7, bucket_size=b)
        t.build(keys.cuda(), None if scheme == "bcht_set" else vals.cuda())
        assert _check(G, t, scheme, keys, vals)["last_build_small"] == int(n == most)


def test_stats_say_which_kernels_ran(G):
    """The find that answers, for default and named shapes; the one-block build; and the looks for
    a victim of long chains, which are no bucket visits: counted where there are any."""
    n = 3000
    keys, vals = W.make_keys(n, 1).cuda(), W.make_values(n, 1).cuda()
    for scheme, cfg, line in (("bcht", {}, 1), ("bcht", {"tile_lanes": 4, "keys_per_lane": 2}, 1),
                              ("bcht", {"keys_per_lane": 1}, 0), ("bcht", {"tile_lanes": 8}, 0),
                              ("bcht", {"find_async": -1}, 0), ("bcht", {"find_async": 1}, 0),
                              ("bcht", {"bucket_size": 32}, 0), ("p2bht", {}, 1), ("iht", {}, 1), ("bcht_lb", {}, 1),
                              ("cuckoo1", {}, 0), ("bcht_set", {}, 1)):
        t = G.HashTable(scheme, n, 0.6, seed=2, **cfg)
        t.build(keys, vals)
        assert t.stats()["find_line"] == line and t.stats()["last_build_small"] == (scheme != "cuckoo1")
        t.build(keys[:100], vals[:100])
    b = G.Batch([n], [0.9], seed=1, tile_lanes=8)
    assert b.table_stats(0)["find_line"] == 0
    n = 1 << 20
    keys, vals = W.make_keys(n, 2).cuda(), W.make_values(n, 2).cuda()
    for lf, some in ((0.99, True), (0.5, False)):
        t = G.HashTable("bcht", n, lf, seed=3, count_probes=1)
        t.build(keys, vals)
        st = t.stats()
        assert (st["victim_looks"] > 0) == some
        assert st["victim_looks"] <= st["insert_evictions"] and st["last_build_small"] == 0


# 3648 warps of three blocks, 2432 of two on 152 SMs: around one chunk of 32 keys a warp, around
# 32, and past it, where the last quarter is claimed
@pytest.mark.parametrize("n", [33, 116737, 3735553, 5000011])
@pytest.mark.parametrize("scheme,lf", [("bcht", 0.95), ("p2bht", 0.75), ("iht", 0.8), ("bcht_lb", 0.9), ("bcht_set", 0.95)])
def test_insert_of_every_key(G, scheme, lf, n):
    """The insert in input order, which serves builds without scratch."""
    keys, vals = W.make_keys(n, n & 0xFFF), W.make_values(n, 3)
    t = G.HashTable(scheme, n, lf, seed=n, group_build=-1, ranked_build=-1)
    t.build(keys.cuda(), None if scheme == "bcht_set" else vals.cuda())
    st = _check(G, t, scheme, keys, vals)
    assert (st["last_build_ranked"], st["last_build_grouped"], st["last_build_small"]) == (0, 0, 0)


@pytest.mark.parametrize("scheme,lf", [("p2bht", 0.78), ("iht", 0.8), ("bcht_lb", 0.95), ("cuckoo1", 0.7), ("bcht", 0.95)])
def test_two_phase_build_from_pageable_arrays(G, scheme, lf):
    """On request, pageable arrays are placed chunk by chunk as they arrive."""
    n = 300007
    keys, vals = W.make_keys(n, 8), W.make_values(n, 8)
    t = G.HashTable(scheme, n, lf, seed=6, ranked_build=1)
    t.build(keys, vals)
    st = _check(G, t, scheme, keys, vals)
    assert (st["last_build_ranked"], st["last_build_grouped"]) == (1, 0) and st["last_h2d_bytes"] == 8 * n


@pytest.mark.parametrize("scheme,lf", [("p2bht", 0.75), ("iht", 0.75), ("bcht_lb", 0.9), ("cuckoo1", 0.7)])
def test_two_phase_build_from_pageable_arrays_of_two_chunks(G, scheme, lf):
    n = (1 << 25) + 1001
    keys, vals = W.make_keys(n, 9), W.make_values(n, 9)
    t = G.HashTable(scheme, n, lf, seed=6, ranked_build=1)
    t.build(keys, vals)
    assert t.stats()["last_build_ranked"] == 1 and t.stats()["n_stored"] == n
    assert torch.equal(t.find(keys.cuda()), vals.cuda())
    absent = W.make_negatives(n, 1 << 20, 9).cuda()
    assert (t.find(absent) == -1).all()


@pytest.mark.parametrize("scheme,n,ranked", [("p2bht", 40001, 0), ("p2bht", 700001, 0), ("p2bht", 40001, -1), ("iht", 40001, -1),
                                             ("iht", 40001, 0)])
def test_schemes_without_evictions_fail_full_tables(G, scheme, n, ranked):
    """At load factor 1 some key finds all its candidates full, in the placement by load as in the
    inserts: every attempt is made, the call says so, and the same table then builds fewer keys."""
    keys, vals = W.make_keys(n, 2), W.make_values(n, 2)
    t = G.HashTable(scheme, n, 1.0, seed=4, max_attempts=3, ranked_build=ranked, group_build=-1 if ranked else 0)
    with pytest.raises(G.GhtError) as e:
        t.build(keys.cuda(), vals.cuda())
    assert e.value.status == "GHT_ERR_BUILD_FAILED"
    assert t.stats()["attempts"] == 3 and t.stats()["built"] == 0
    most = n // 2
    t.build(keys[:most].cuda(), vals[:most].cuda())
    st = _check(G, t, scheme, keys[:most], vals[:most])
    assert st["last_build_ranked"] == (1 if ranked == 0 else 0) and st["attempts"] == 1


def test_load_balanced_overflow_beyond_the_list(G):
    """Keys whose candidates all lie in an eighth of the buckets under the first constants: the
    placement by load overflows its list, the attempt is redone with the insert of every key, which
    cannot hold them either, and the next constants build the table."""
    n, lf, seed = 40000, 0.8, 13
    m = O.num_buckets(n, lf, 16)
    a, c = O.derive_constants(seed, 0, 3)
    cand = np.arange(1, 1 << 25, dtype=np.uint64)
    for i in range(3):
        h = ((np.uint64(a[i]) * cand + np.uint64(c[i])) % np.uint64(O.PRIME)) % np.uint64(m)
        cand = cand[h < m // 8]
    crowd = cand[:n].astype(np.uint32)
    assert crowd.size == n
    keys, vals = torch.from_numpy(crowd.view(np.int32).copy()), W.make_values(n, 5)
    t = G.HashTable("bcht_lb", n, lf, seed=seed)
    t.build(keys.cuda(), vals.cuda())
    st = _check(G, t, "bcht_lb", keys, vals)
    assert st["attempts"] == 2 and st["last_build_ranked"] == 1


@pytest.mark.parametrize("n", [3000, 60001])
@pytest.mark.parametrize("threshold", [1, 2, 16, 17])
def test_iht_thresholds_at_the_ends(G, threshold, n):
    """From a primary that takes no key at first to one that takes a full bucket, in one block and
    over the whole device."""
    keys, vals = W.make_keys(n, 3), W.make_values(n, 3)
    t = G.HashTable("iht", n, 0.5, seed=2, threshold=threshold)
    t.build(keys.cuda(), vals.cuda())
    st = _check(G, t, "iht", keys, vals)
    assert st["last_build_small"] == (n == 3000) and st["threshold"] == threshold


@pytest.mark.parametrize("n,two_phase", [(6000000, 1), (5999999, 0), (1000, 0)])
def test_few_keys_in_a_large_table_of_bucket_size_one(G, n, two_phase):
    keys, vals = W.make_keys(n, 4), W.make_values(n, 4)
    t = G.HashTable("cuckoo1", 1 << 24, 0.8, seed=2)
    t.build(keys.cuda(), vals.cuda())
    st = t.stats()
    assert (st["last_build_ranked"], st["last_build_grouped"], st["n_stored"]) == (two_phase, two_phase, n)
    q = W.make_queries(keys, 1 << 20, 0.5, seed=3)
    assert (O._u32(t.find(q.cuda()).cpu()) == O.lookup(keys, vals, q)).all()
