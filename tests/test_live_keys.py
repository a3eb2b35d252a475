"""Which keys the producers of an attention kernel may read before earlier work of the stream is complete: planned by the
library's host side, recorded without a GPU."""
import pytest

from tests import host_plan as hp

A, B, C = 0x100, 0x200, 0x300


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return hp.build(tmp_path_factory.mktemp("hostplan"))


@pytest.fixture
def kv(lib):
    h = hp.Handle(lib)
    h.alloc(0, 1, 2, 3)
    for t in range(4):
        assert h.append({t: 1000 + t}, A) == 0
    yield h
    h.close()


def test_keys_of_the_last_append_of_a_stream_are_live(kv):
    assert kv.append({0: 5, 1: 1}, A) == 0
    assert kv.live([(0, 1, 1005), (1, 1, 1002), (2, 1, 1002)], A) == {0: 992, 1: 992, 2: hp.INT_MAX}
    assert kv.append({2: 1}, A) == 0                           # waits for the append before it
    assert kv.live([(0, 1, 1005), (2, 1, 1003)], A) == {0: hp.INT_MAX, 2: 992}


@pytest.mark.parametrize("later", ["appends", "moves"])
def test_writers_of_another_stream_leave_the_keys_of_this_one_live(kv, later):
    assert kv.append({0: 7}, B) == 0
    for t in (1, 2, 1):
        assert (kv.append({t: 3}, A) if later == "appends" else kv.prune(t, 100, 110, A)) == 0
    assert kv.live([(0, 1, 1007)], B) == {0: 992}
    assert kv.live([(0, 1, 1007)], B) == {0: 992}              # reading changes nothing
    assert kv.append({3: 1}, B) == 0                           # the next writer of B has waited
    assert kv.live([(0, 1, 1007)], B) == {0: hp.INT_MAX}


def test_a_task_written_on_two_streams(kv):
    assert kv.append({0: 100}, B) == 0                         # keys from 1000 on
    assert kv.live([(0, 1, 1100)], A) == {0: 992}              # whoever reads them on A has ordered the streams; live all the same
    assert kv.append({0: 1}, A) == 0
    assert kv.live([(0, 1, 1101)], A) == {0: 1088}
    assert kv.live([(0, 1, 1101)], B) == {0: 992}
    assert kv.append({1: 1}, A) == 0
    assert kv.live([(0, 1, 1101)], A) == {0: hp.INT_MAX}
    assert kv.live([(0, 1, 1101)], B) == {0: 992}


def test_more_streams_than_are_kept(kv):
    streams = [0x1000 * i for i in range(1, 40)]
    for s in streams:
        assert kv.append({0: 1}, s) == 0
    assert kv.live([(1, 1, 1001)], streams[0]) == {1: 0}       # forgotten: nothing is read ahead
    assert kv.live([(1, 1, 1001)], streams[-1]) == {1: hp.INT_MAX}
    assert kv.append({1: 1}, streams[0]) == 0
    assert kv.live([(1, 1, 1002)], streams[0]) == {1: 992}


def test_a_series_of_moves(kv):
    assert kv.prune(0, 64, 100, A) == 0 and kv.prune(1, 33, 34, A) == 0
    n0, n1 = 1000 - 36, 1000
    assert kv.live([(0, 1, n0), (1, 1, n1)], A) == {0: 64, 1: 32}
    assert kv.prune(2, 64, 100, A) == 0                        # an attention call came between: a series of its own
    assert kv.live([(0, 1, n0), (1, 1, n1), (2, 1, 1002 - 36)], A) == {0: hp.INT_MAX, 1: hp.INT_MAX, 2: 64}
