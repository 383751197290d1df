"""Batched tables on the paths beside the default one: a crowded table beside
others, every find shape, and the memory a batch takes."""

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


@pytest.mark.parametrize("run", [True, False])
def test_a_crowded_table_costs_no_table_its_attempt(G, run):
    """All keys of one table share their first bucket, so they fill the batch's overflow list and
    other tables' keys find it full; every table's first constants build it (the oracle's insert of
    the crowded one too), so a batch with a single attempt must build them all."""
    n, others, seed = 6000, 40, 29
    m = O.num_buckets(n, 0.5, 16)
    a, c = O.derive_constants(seed, 0, 3)
    cand = np.arange(1, 1 << 24, dtype=np.uint64)
    h0 = ((np.uint64(a[0]) * cand + np.uint64(c[0])) % np.uint64(O.PRIME)) % np.uint64(m)
    crowd = cand[h0 == h0[0]][:n].astype(np.uint32)
    alone = O.Table(O.BCHT, n, 0.5)
    alone.set_constants(a, c)
    rest = W.make_keys(2 * others * 300, 3).numpy().view(np.uint32)
    rest = rest[~np.isin(rest, crowd)][: others * 300]
    keys = torch.from_numpy(np.concatenate([crowd, rest]).view(np.int32).copy())
    vals = W.make_values(keys.numel(), 8)
    assert alone.build(keys[:n], vals[:n]) == 1
    b = G.Batch([n] + [300] * others, [0.5] + [0.95] * others, seed=seed, max_attempts=1)
    offs = np.concatenate([[0], n + 300 * np.arange(others + 1)]).astype(np.uint64)
    b.set_layout(offs, offs)
    dk, dv = keys.cuda(), vals.cuda()
    for _ in range(3):
        if run:
            out = b.run(dk, dv, dk)
        else:
            b.build(dk, dv)
            out = b.find(dk)
        assert torch.equal(out, dv)
        st = b.stats()
        assert st["tables_failed"] == 0 and st["rebuilds"] == 0
        assert all(b.table_stats(t)["attempts"] == 1 for t in range(others + 1))


def _uneven(seed):
    return W.make_batch(60, 3, 13, 0.8, 0.99, 2.0, 0.6, seed=seed)


@pytest.mark.parametrize("cfg,shape", [
    ({}, (4, 2, 1)), ({"tile_lanes": 4, "keys_per_lane": 2}, (4, 2, 1)), ({"find_async": -1}, (4, 2, 0)),
    ({"tile_lanes": 8}, (8, 2, 0)), ({"tile_lanes": 16}, (16, 2, 0)), ({"keys_per_lane": 1}, (4, 1, 0)),
    ({"tile_lanes": 8, "keys_per_lane": 1}, (8, 1, 0)), ({"tile_lanes": 16, "keys_per_lane": 1}, (16, 1, 0)),
    ({"tile_lanes": 4, "keys_per_lane": 6}, (4, 6, 0))])
def test_every_batch_find_shape(G, cfg, shape):
    """A config's shape is the one that runs (a missing half is the default's), the default and the
    values of the default config are the line find, and all answer alike; sentinel queries too."""
    w = _uneven(5)
    b = G.Batch(w["capacities"], w["load_factors"], seed=2, **cfg)
    st = b.stats()
    assert (st["tile_lanes"], st["keys_per_lane"], st["find_line"]) == shape
    b.set_layout(w["key_offsets"], w["query_offsets"])
    q = w["queries"].clone()
    q[5::37] = -1
    b.build(w["keys"].cuda(), w["values"].cuda())
    got = O._u32(b.find(q.cuda()).cpu())
    ko, qo = w["key_offsets"], w["query_offsets"]
    for t in range(b.num_tables):
        want = O.lookup(w["keys"][ko[t]:ko[t + 1]], w["values"][ko[t]:ko[t + 1]], q[qo[t]:qo[t + 1]])
        assert (got[qo[t]:qo[t + 1]] == want).all(), t


@pytest.mark.parametrize("cfg", [{"keys_per_lane": 1}, {"find_async": -1}, {"tile_lanes": 16}, {"tile_lanes": 4, "keys_per_lane": 2}])
def test_pool_find_shapes_answer_alike(G, cfg):
    pool = G.Pool(1 << 28, **cfg)
    k, v = W.make_keys(30000, 1), W.make_values(30000, 1)
    ticket, tid = pool.submit_build(30000, 0.95, 1, k.cuda(), v.cuda())
    assert pool.wait(ticket)["status"] == 0
    for n in (1, 33, 70001):
        q = W.make_queries(k, n, 0.6, seed=n)
        d = q.cuda()
        out = torch.empty_like(d)
        torch.cuda.synchronize()
        assert pool.wait(pool.submit_find(tid, d, out))["status"] == 0
        assert (O._u32(out.cpu()) == O.lookup(k, v, q)).all()
    pool.close()


def test_a_batch_takes_placement_scratch_only_where_it_places(G):
    """An insert shape without the placement keeps no scratch for it; the autotuner takes it to
    time the default shape and keeps it only if that wins."""
    n = 1 << 24
    slots = O.num_buckets(n, 0.9, 16) * 128
    scratch = (slots // 128 + 3 * (n // 4)) * 4  # 55 MB
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]

    def taken():
        torch.cuda.synchronize()
        return before - torch.cuda.mem_get_info()[0] - slots

    b = G.Batch([n], [0.9], seed=1, build_tile_lanes=8)
    assert taken() < scratch // 2
    b.close()
    b = G.Batch([n], [0.9], seed=1)
    assert taken() > scratch // 2
    b.close()
    assert taken() + slots < scratch // 2

    w = _uneven(9)
    k, v, q = w["keys"].cuda(), w["values"].cuda(), w["queries"].cuda()
    for cfg in ({"build_tile_lanes": 8}, {}):
        b = G.Batch(w["capacities"], w["load_factors"], seed=4, **cfg)
        b.set_layout(w["key_offsets"], w["query_offsets"])
        first = b.run(k, v, q)
        b.autotune(k, v, q)
        assert torch.equal(b.run(k, v, q), first)
