"""What the library's host side plans and launches, recorded without a GPU."""
import pytest

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
