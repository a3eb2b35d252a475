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


def test_a_forked_child_is_live_as_a_whole(kv):
    """Its page-table row and the copy of its last page are written by the launches in front."""
    kv.alloc(9)
    assert kv.append({9: 1}, A) == 0                           # nothing of the parent is in flight any more
    assert kv.fork(0, 5, A) == 0
    assert kv.live([(5, 1, 1000), (0, 1, 1000)], A) == {5: 0, 0: hp.INT_MAX}
    assert kv.append({5: 1}, A) == 0
    assert kv.live([(5, 1, 1001), (0, 1, 1000)], A) == {5: 992, 0: hp.INT_MAX}


@pytest.mark.parametrize("D", [64, 128])
def test_a_shared_range_is_as_live_as_the_row_it_is_read_through(lib, D):
    kv = hp.Handle(lib, D=D, Hq=8, Hkv=2)
    kv.tune(2, 0)                                              # groups however little they save
    kv.alloc(0)
    assert kv.append({0: 1003}, A) == 0
    for c in range(1, 8):
        assert kv.fork(0, c, A) == 0
    kv.forget()
    assert kv.attend([(c, 1, 1003) for c in (7, 6, 5, 4, 3, 2, 1, 0)], A) == 0
    found = {}
    for l in kv.launches():
        if l["kind"] in (hp.DECODE, hp.UMMA) and l["run_ahead"]:
            for s in l["segs"]:
                found.setdefault("own" if s["causal"] else "shared", []).append(s["live_from"])
    assert found["shared"] == [0]
    kv.close()


def test_extended_tasks_are_live_from_their_last_page_on(kv):
    """A page that the growth replaces by a private copy, and new entries of the page table, are being written."""
    assert kv.fork(0, 5, A) == 0 and kv.fork(0, 6, A) == 0
    assert kv.truncate(6, 500) == 0                            # inside a page that the others hold
    assert kv.append({1: 1}, A) == 0
    assert kv.extend({6: 1, 2: 40}, A) == 0
    assert kv.live([(6, 1, 500), (2, 1, 1002), (5, 1, 1000)], A) == {6: 496, 2: 992, 5: hp.INT_MAX}


def test_growth_that_tells_the_device_nothing_leaves_everything_live(kv):
    assert kv.append({1: 5}, A) == 0
    kv.forget()
    assert kv.extend({0: 1}, A) == 0 and kv.launches() == []   # inside its last page
    assert kv.append({0: 0, 2: 0}, A) == 0 and kv.launches() == []
    assert kv.truncate(2, 0) == 0 and kv.fork(2, 5, A) == 0 and kv.launches() == []
    assert kv.live([(1, 1, 1006)], A) == {1: 992}


def test_a_step_that_has_begun(kv):
    assert kv.fork(0, 6, A) == 0 and kv.truncate(6, 500) == 0
    assert kv.append({1: 1}, A) == 0
    assert kv.step_begin([(6, 1, 501), (2, 40, 1042)], A) == 0
    assert kv.live([(6, 1, 500), (2, 1, 1002), (3, 1, 1003)], A) == {6: 496, 2: 992, 3: hp.INT_MAX}
    kv.forget()
    assert kv.step_layer(0, A) == 0                            # behind its own append, which waits for all that
    launches = [l for l in kv.launches() if l["kind"] in (hp.DECODE, hp.UMMA)]
    assert [(l["kind"], l["run_ahead"], l["overlapped"]) for l in launches] == [(hp.UMMA, 1, 0), (hp.DECODE, 0, 1)]
    live = {s["task"]: s["live_from"] for l in launches for s in l["segs"]}
    assert live == {6: 500, 2: 1002}


def test_a_prune_that_goes_through_the_staging_area(kv):
    assert kv.fork(0, 5, A) == 0
    assert kv.append({1: 1}, A) == 0
    assert kv.prune(5, 100, 300, A) == 0                       # shares its pages: a new table row, a copied page, an append
    assert kv.live([(5, 1, 800), (0, 1, 1000)], A) == {5: 96, 0: hp.INT_MAX}


@pytest.fixture
def layered(lib):
    h = hp.Handle(lib, layers=3)
    h.alloc(0, 1, 2, 3)
    for t in range(4):
        assert h.append({t: 1000 + t}, A) == 0
    yield h
    h.close()


def writer(kv, which, stream):
    assert {"fork": lambda: kv.fork(1, 5, stream), "write": lambda: kv.write(1, {2: 20}, stream)}[which]() == 0


# one query (the decode kernel) and 40 (the tcgen05 kernel)
@pytest.mark.parametrize("queries", [1, 40])
@pytest.mark.parametrize("which", ["fork", "write"])
def test_rows_that_a_decode_launch_writes_are_live(layered, which, queries):
    """A step of decode rows: the layers' attention launches write the step's rows, and let the next launch start before.  A
    writer between the begin of the step and a layer changes nothing about that."""
    kv = layered
    assert kv.step_begin([(0, 1, 1001)], A) == 0
    writer(kv, which, A)
    kv.forget()
    assert kv.step_layer(0, A) == 0
    assert [(l["kind"], l["writes"]) for l in kv.launches()] == [(hp.DECODE, 1)]
    assert kv.live([(0, queries, 1001)], A) == {0: 992}
    assert kv.step_layer(1, A) == 0
    writer(kv, "write", A)                                     # waits for the layers: their rows are complete, its own are not
    assert kv.live([(0, queries, 1001), (2, queries, 1002)], A) == {0: hp.INT_MAX, 2: 976}
    assert kv.step_layer(2, A) == 0
    assert kv.live([(0, queries, 1001), (2, queries, 1002)], A) == {0: 992, 2: hp.INT_MAX}


@pytest.mark.parametrize("queries", [1, 40])
def test_rows_that_a_decode_launch_writes_are_live_on_its_own_stream(layered, queries):
    kv = layered
    assert kv.step_begin([(0, 1, 1001), (1, 1, 1002)], A) == 0
    for l in range(3):
        assert kv.step_layer(l, B) == 0
    assert kv.append({2: 1}, A) == 0                           # says nothing about B
    assert kv.live([(0, queries, 1001), (1, queries, 1002)], B) == {0: 992, 1: 992}
    assert kv.append({3: 1}, B) == 0
    assert kv.live([(0, queries, 1001), (1, queries, 1002)], B) == {0: hp.INT_MAX, 1: hp.INT_MAX}


def test_layers_run_ahead_behind_a_layer(layered):
    """Not behind the begin of the step or a writer, whose keys the step's plan does not know; again behind the layer behind it."""
    kv = layered
    assert kv.step_begin([(0, 1, 1001), (2, 1, 1003)], A) == 0
    ahead = []

    def layer(l, stream=A):
        kv.forget()
        assert kv.step_layer(l, stream) == 0
        (launch,) = kv.launches()
        assert launch["kind"] == hp.DECODE and launch["writes"] == 1
        assert {s["task"]: s["live_from"] for s in launch["segs"]} == {0: 1000, 2: 1002}
        ahead.append(launch["run_ahead"])

    layer(0), layer(1), layer(2)
    assert kv.attend([(1, 1, 1001)], A) == 0                   # a reader
    layer(0)
    writer(kv, "write", A)
    layer(1), layer(2)
    writer(kv, "fork", B)                                      # of whatever stream
    layer(0), layer(1)
    layer(2, B), layer(0, B)                                   # another stream: its first layer is not behind a layer
    assert ahead == [0, 1, 1, 1, 0, 1, 0, 1, 0, 1]
