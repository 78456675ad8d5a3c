"""Server.submit_group takes every kind of entry that unpacks into six fields, and
whatever it queues keeps its buffers referenced until the group has finished.
The library is a stand-in: no device."""
from collections import deque

import numpy as np
import pytest

from paper_2007_10752_gb300 import tdes


class _Lib:
    """Records the descriptors a group queues."""

    def __init__(self):
        self.queued = []

    def tdes_server_submit_group(self, handle, addr, n, ticket):
        self.queued += [tdes.Desc.from_buffer_copy(d) for d in (tdes.Desc * n).from_address(addr)]
        ticket._obj.value = 7
        return tdes.TDES_OK

    def tdes_server_poll_group(self, handle, ticket, n, statuses):
        return 0


@pytest.fixture
def server(monkeypatch):
    lib = _Lib()
    monkeypatch.setattr(tdes, "load", lambda *a: lib)
    s = tdes.Server.__new__(tdes.Server)
    s.handle, s._keep, s._submits, s.lib = 1, {}, 0, lib
    yield s
    s.handle = None  # nothing for close() to destroy


@pytest.mark.parametrize("kind", [tuple, list, deque, iter, np.array, "unpacks_only"], ids=str)
def test_entry_kinds(server, kind):
    x, y = np.zeros(8, np.uint8), np.zeros(8, np.uint8)

    class Unpacks:
        def __init__(self, fields):
            self.fields = fields

        def __iter__(self):
            return iter(self.fields)

    fields = (0, 3, 5, x, y, 8)
    make = {"unpacks_only": Unpacks, np.array: lambda f: np.array(f, dtype=object)}.get(kind, kind)
    assert server.submit_group([make(fields)]) == (7, 1)
    (d,) = server.lib.queued
    assert (d.mode, d.key_index, d.nbytes) == (0, 3, 8)
    count, kept = server._keep[7]
    assert count == 1 and [id(b) for b in kept] == [id(x), id(y)]
    server.poll_group((7, 1))
    assert 7 not in server._keep


@pytest.mark.parametrize("bad", [(0, 3, 5, 8, 16), deque((0, 3, 5, 8, 16, 8, 9)), 5], ids=str)
def test_nothing_is_queued_for_an_entry_that_is_refused(server, bad):
    with pytest.raises((ValueError, TypeError)):
        server.submit_group([(0, 3, 5, 8, 16, 8), bad])
    assert server.lib.queued == [] and server._keep == {}


def test_plain_addresses_are_the_callers(server):
    assert server.submit_group([(0, 3, 5, 64, 128, 8)] * 3) == (7, 3)
    assert len(server.lib.queued) == 3 and server._keep == {}
