"""Builds and finds at the sizes where the kernels' splits of the work change:
around a warp's chunk, around one share per warp, and past it."""

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
                                         ("iht", 0.8, 3735553), ("p2bht", 0.75, 5000011)])
def test_insert_shares(G, scheme, lf, n):
    _check(G, scheme, n, lf, seed=n & 0xFFFF)
