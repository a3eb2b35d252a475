"""What the library's host side plans and launches, recorded without a GPU."""
import pytest

from paper_2608_10402_b200 import tide
from tests import host_plan as hp


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return hp.build(tmp_path_factory.mktemp("hostplan"))


@pytest.mark.parametrize("caps,kinds", [((0, 400, 4000, 0, 2048), [hp.TILE]), ((0, 400, 0, 0, 2048), [hp.TILE]), ((0, 400, 10, 80000, 2048), [hp.TILE]),
                                        ((0, 0, 4000, 80000, 2048), [hp.UMMA, hp.MERGE]), ((8, 400, 4000, 80000, 2048), [hp.UMMA, hp.MERGE])])
def test_fixed_launch_shapes_take_the_warp_tiles_where_only_these_fit(lib, caps, kinds):
    """64-wide heads: a row of 2000 tokens is 250 warp-MMA tiles, which are not cut, or 64 tcgen05 items, which are cut along
    the keys and merged.  Shapes that hold either plan are accepted."""
    kv = hp.Handle(lib, Hq=8, Hkv=2, D=64)
    kv.alloc(0)
    assert kv.append({0: 9000}) == 0
    assert kv.fix_grids(*caps) == 0
    assert kv.step_begin([(0, 2000, 11000)]) == 0
    kv.forget()
    assert kv.step_layer(0) == 0
    assert [l["kind"] for l in kv.launches() if l["segs"]] == kinds
    plan = kv.plan()
    assert (plan["merge_rows"] == 0) == (kinds == [hp.TILE]) and plan["prefill_items"] <= max(caps[1], caps[2])
    kv.close()


def test_fixed_launch_shapes_that_hold_neither_plan_are_refused(lib):
    kv = hp.Handle(lib, Hq=8, Hkv=2, D=64)
    kv.alloc(0)
    assert kv.append({0: 9000}) == 0
    for caps in ((0, 200, 10, 80000, 2048), (0, 200, 4000, 0, 2048), (0, 400, 4000, 0, 1999)):
        assert kv.fix_grids(*caps) == 0
        assert kv.step_begin([(0, 2000, 11000)]) == -8
        assert kv.attend([(0, 1, 9000)]) == 0 and kv.attend([(0, 1, 9001)]) == -7      # nothing has changed
    kv.close()


@pytest.mark.parametrize("geom", [(28, 4, 128, 16), (16, 1, 64, 32)])
@pytest.mark.parametrize("groups", [1, 2, 4, 7])
def test_a_host_step_is_cut_between_and_inside_rows(lib, geom, groups):
    """Every token of every row is attended once, in order, its context ending with it; long rows are cut between groups at
    whole tcgen05 items; the groups take turns on two streams, each behind its own append."""
    kv = hp.Handle(lib, *geom)
    kv.tune(tide.TUNE_HOST_STEP_CHUNKS, groups)
    kv.tune(tide.TUNE_HOST_ZERO_COPY, 0)
    prefix, new = [0, 700, 15, 2500, 3000, 1, 64, 900], [1400, 1, 1, 1, 733, 1, 160, 17]
    kv.alloc(*range(8))
    assert kv.append(dict(enumerate(prefix))) == 0
    kv.forget()
    assert kv.step_host([(t, n, p + n) for t, (p, n) in enumerate(zip(prefix, new))]) == 0
    launches = kv.launches()
    appends = [l for l in launches if l["kind"] == hp.APPEND]
    assert sum(l["items"] for l in appends) == sum(new) and (groups == 1) == (len(appends) == 1) and len(appends) <= groups
    if groups > 1:
        assert all(a["stream"] != b["stream"] for a, b in zip(appends, appends[1:])) and {a["stream"] for a in appends} == {a["stream"] for a in appends[:2]}
    seen, parts, stream = dict(enumerate(prefix)), dict.fromkeys(range(8), 0), None
    for l in launches:
        if l["kind"] == hp.APPEND:
            stream = l["stream"]
        if l["kind"] in (hp.DECODE, hp.UMMA):
            assert l["stream"] == stream
            for s in l["segs"]:
                assert s["p"] == seen[s["task"]]
                seen[s["task"]] += s["n"]
                parts[s["task"]] += 1
    assert seen == {t: p + n for t, (p, n) in enumerate(zip(prefix, new))}
    assert (parts[0] > 1) == (groups > 1) and all(parts[t] == 1 for t in (1, 2, 3, 5, 7))
    kv.close()


def test_only_an_answer_that_has_landed_is_a_work_item(lib):
    """The place of the answer holds an older item, or nothing at all, until the hardware has written it."""
    for stale in (-1, 0, 7, 99, 100, 2 ** 31 - 1, -2 ** 31):
        assert lib.claimed(0, stale, 100) == -1
    assert [lib.claimed(1, x, 100) for x in (-1, 0, 99, 100, 2 ** 31 - 1)] == [-1, 0, 99, -1, -1]


@pytest.mark.parametrize("Hq,Hkv", [(16, 16), (28, 4)])
def test_rows_that_the_results_overwrite_are_appended_first(lib, Hq, Hkv):
    """A caller may have a layer's results written over its new K/V rows.  Attention blocks that write the rows of their own items
    would read rows that other blocks' results have replaced, so such a layer has its append in front."""
    kv = hp.Handle(lib, Hq=Hq, Hkv=Hkv, layers=2)
    tasks, T = (0, 1, 2), 3
    kv.alloc(*tasks)
    assert kv.append({t: 100 for t in tasks}) == 0
    assert kv.step_begin([(t, 1, 101) for t in tasks]) == 0
    k, o, lse = T * Hkv * 128 * 2, T * Hq * 128 * 2, T * Hq * 4

    def kinds(**where):
        kv.forget()
        assert kv.step_layer(0, **where) == 0
        return [(l["kind"], l["writes"], l["run_ahead"]) for l in kv.launches()]

    apart, behind = [(hp.DECODE, 1, 1)], [(hp.APPEND, 1, 0), (hp.DECODE, 0, 1)]
    K, V, O, X = 1 << 30, 2 << 30, 4 << 30, 5 << 30
    assert kinds(lse=X) == [(hp.DECODE, 1, 0)]                 # the first layer waits
    for rows in (K, V):
        assert kinds(out=rows) == behind and kinds(out=rows + k - 16) == behind and kinds(out=rows - o + 16) == behind
        assert kinds(lse=rows + k - 4) == behind and kinds(lse=rows - lse + 4) == behind
        assert kinds(out=rows + k) == apart and kinds(out=rows - o) == apart
        assert kinds(lse=rows + k) == apart and kinds(lse=rows - lse) == apart
    assert kinds(q=O) == apart                                 # results over the queries, as ever
    kv.close()


@pytest.mark.parametrize("D", [64, 128])
def test_which_steps_write_their_rows_in_the_decode_launch(lib, D):
    """One token a row, or up to 1.25 MiB of new K and V; only decode-style rows, no groups, no fixed launch shapes."""
    kv = hp.Handle(lib, Hq=16, Hkv=16, D=D, max_rows=400, max_tasks=400, num_pages=16384)
    kv.alloc(*range(360))
    assert kv.append({t: 100 for t in range(360)}) == 0
    length = [100] * 400

    def kinds(new):
        rows = [(t, c, length[t] + c) for t, c in new.items()]
        assert kv.step_begin(rows) == 0
        for t, c in new.items():
            length[t] += c
        kv.forget()
        assert kv.step_layer(0) == 0
        return [(l["kind"], l["writes"]) for l in kv.launches()]

    one, two = [(hp.DECODE, 1)], [(hp.APPEND, 1), (hp.DECODE, 0)]
    most = (5 << 18) // (16 * D * 4)                           # tokens: 160, 320
    assert kinds({t: 1 for t in range(360)}) == one            # beyond it, but one each
    assert kinds({t: 16 for t in range(most // 16)}) == one
    assert kinds({t: 16 for t in range(most // 16)} | {350: 1}) == two
    assert kinds({t: 1 for t in range(most - 2)} | {350: 2}) == one
    assert kinds({t: 1 for t in range(most - 1)} | {350: 2}) == two
    assert kinds({0: 1, 1: 17}) == [(hp.APPEND, 1), (hp.UMMA, 0), (hp.DECODE, 0)]       # a resume row
    assert kv.fix_grids(4096, 0, 0, 0, 4096) == 0
    assert kinds({0: 1, 1: 1}) == two
    assert kv.fix_grids(0, 0, 0, 0, 0) == 0
    assert kinds({0: 1, 1: 1}) == one
    kv.alloc(390)
    assert kv.append({390: 600}) == 0 and kv.fork(390, 391) == 0 and kv.fork(390, 392) == 0
    length[390:393] = [600] * 3
    assert kinds({390: 1, 391: 1, 392: 1}) == one              # a group would not save enough
    kv.tune(tide.TUNE_MIN_SAVED_BYTES, 0)
    assert kinds({390: 1, 391: 1, 392: 1}) == [(hp.APPEND, 1), (hp.DECODE, 0), (hp.MERGE, 0)]
    kv.close()


@pytest.mark.parametrize("D", [64, 128])
def test_large_layers_of_64_wide_heads_append_first(lib, D):
    """Up to 1.5 GiB of K and V: 393216 tokens of 16 heads of 64."""
    kv = hp.Handle(lib, Hq=16, Hkv=16, D=D, max_rows=8, num_pages=32768, max_pages=4100)
    kv.alloc(*range(7))
    for t in range(6):
        assert kv.append({t: 65534}) == 0
    assert kv.append({6: 5}) == 0

    def kinds(rows):
        assert kv.step_begin(rows) == 0
        kv.forget()
        assert kv.step_layer(0) == 0
        return [(l["kind"], l["writes"]) for l in kv.launches()]

    one, two = [(hp.DECODE, 1)], [(hp.APPEND, 1), (hp.DECODE, 0)]
    assert kinds([(t, 1, 65535) for t in range(6)]) == one
    assert kinds([(t, 1, 65536) for t in range(6)]) == one     # 6 * 65536 = 393216
    assert kinds([(t, 1, 65537) for t in range(5)] + [(6, 1, 6)]) == one
    assert kinds([(t, 1, 65538) for t in range(5)] + [(5, 1, 65537)]) == (two if D == 64 else one)
    kv.close()
