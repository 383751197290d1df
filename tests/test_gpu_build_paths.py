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
    T = O.Table(O.BCHT if sets else G.SCHEMES[scheme], keys.numel(), 0.5, b=st["bucket_size"], m=st["num_buckets"])
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
