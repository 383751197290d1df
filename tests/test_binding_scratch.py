"""The binding's scratch tensors on CPU, with the library's calls replaced: a
device without room for a build's scratch."""

import pytest
import torch

from paper_2108_07232_gb300 import _binding as B


@pytest.fixture
def table(monkeypatch):
    """A table object without a handle whose library calls are recorded."""
    calls = []
    t = B.HashTable.__new__(B.HashTable)
    t._t, t.scheme, t.device, t._grouped_find = None, B.BCHT, torch.device("cpu"), True
    t._stream = lambda: None
    t.calls = calls
    t.need, t.room = 1 << 20, 1 << 30
    empty = torch.empty

    def limited(n, *args, **kw):
        if isinstance(n, int) and kw.get("dtype") == torch.uint8 and n > t.room:
            raise torch.OutOfMemoryError("no room")
        return empty(n, *args, **kw)

    monkeypatch.setattr(torch, "empty", limited)
    monkeypatch.setattr(B, "ght_build_scratch_bytes", lambda *a: t.need)
    monkeypatch.setattr(B, "ght_build_scratch_bytes_for", lambda *a: t.need, raising=False)
    monkeypatch.setattr(B, "ght_find_scratch_bytes", lambda *a: t.need)
    monkeypatch.setattr(B, "ght_set_build_scratch", lambda h, p, n: calls.append(("scratch", n)))
    monkeypatch.setattr(B, "ght_build_host", lambda h, k, v, n: calls.append(("build", n)))
    return t


def test_a_build_runs_without_room_for_scratch(table):
    keys = torch.arange(10, dtype=torch.int32)
    table.room = 1000
    table.build(keys, keys)
    assert table.calls == [("build", 10)]
    # with room again the scratch is taken; a larger one that does not fit leaves it in place
    table.room = 1 << 30
    table.build(keys, keys)
    table.need, table.room = 1 << 21, 1 << 20
    table.build(keys, keys)
    assert table.calls == [("build", 10), ("scratch", 1 << 20), ("build", 10), ("build", 10)]
    assert table._scratch_bytes == 1 << 20


def test_a_grouped_find_without_room_still_fails(table):
    table.room = 1000
    with pytest.raises(torch.OutOfMemoryError):
        table._ensure_find_scratch(10)


def test_a_pool_request_keeps_its_tensors_past_a_timeout(monkeypatch):
    """A wait that runs out leaves the request pending, and the device may still use its arrays."""
    answers = [(7, None), (0, 0), (7, None), (1, 1)]  # (return code, status written or none)

    class Lib:
        def ght_pool_submit_find(self, p, t, q, o, n):
            return 5

        def ght_pool_wait(self, p, ticket, timeout, ref):
            rc, status = answers.pop(0)
            if status is not None:
                ref._obj.status = status
            return rc

    monkeypatch.setattr(B, "lib", lambda: Lib())
    monkeypatch.setattr(B, "ght_last_error", lambda: "")
    pool = B.Pool.__new__(B.Pool)
    pool._p, pool._keep = None, {}
    for done in (lambda: pool.wait(5), lambda: pytest.raises(B.GhtError, pool.wait, 5)):
        ticket = pool.submit_find(0, torch.zeros(3, dtype=torch.int32), torch.zeros(3, dtype=torch.int32))
        with pytest.raises(B.GhtError):
            pool.wait(ticket)
        assert ticket in pool._keep
        done()
        assert ticket not in pool._keep


def test_host_arrays_are_asked_for_by_what_they_are(table, monkeypatch):
    """A build that needs no scratch from device arrays may need some from page-locked ones."""
    monkeypatch.setattr(B, "ght_build_scratch_bytes", lambda *a: 0)
    keys = torch.arange(10, dtype=torch.int32)
    table.build(keys, keys)
    assert table.calls == [("scratch", 1 << 20), ("build", 10)]
