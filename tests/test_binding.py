"""Argument marshalling of the CPython module, without a GPU: a NULL handle is refused by the library itself, so a call
that gets that far has converted its arguments."""
import numpy as np
import pytest


@pytest.fixture(scope="module")
def tide():
    from paper_2608_10402_b200 import build
    build.build()
    from paper_2608_10402_b200 import tide as t
    t._prepare_binding()
    return t


@pytest.mark.parametrize("ids,indptr", [([1, 2], [0, 1, 2]), (np.arange(2), np.arange(3)), (np.arange(2, dtype=np.int32), np.arange(3, dtype=np.int32)),
                                        (np.arange(8, dtype=np.int32)[::4], np.arange(3, dtype=np.uint32)), ((), (0,))])
def test_task_lists_of_every_kind(tide, ids, indptr):
    assert tide._b.append(0, ids, indptr, None, 4096, 0) == tide.ERR_INVALID_ARG
    assert tide._b.extend(0, ids, indptr, 0) == tide.ERR_INVALID_ARG
    assert tide._b.write(0, 0, ids, indptr, np.zeros(4), None, 0) == tide.ERR_INVALID_ARG
    with pytest.raises(AssertionError):
        tide._b.append(0, ids, ids, None, None, 0)


def test_pointers_rows_and_numbers(tide):
    import torch
    rows = tide.rows_array([(0, 1, 5), (1, 2, 7)])
    x = torch.zeros(4, dtype=torch.bfloat16)
    assert tide._b.attend(0, 0, rows, None, x, 0.5, x, None, 0) == tide.ERR_INVALID_ARG
    assert tide._b.step_begin(0, rows, 0) == tide.ERR_INVALID_ARG
    assert tide._b.step_layer(0, np.int64(0), x, x, x, 1, x, np.zeros(2, np.float32), 0) == tide.ERR_INVALID_ARG
    assert tide._b.step_host(0, rows, x, x, x, 0.5, x, None, 0) == tide.ERR_INVALID_ARG
    assert tide._b.truncate(0, np.int32(3), 2) == tide.ERR_INVALID_ARG
    assert tide._b.prune(0, 1, 2, 3, 0) == tide.ERR_INVALID_ARG
    for bad in (lambda: tide._b.truncate(0, 1.5, 2), lambda: tide._b.attend(0, 0, object(), None, x, 0.5, x, None, 0),
                lambda: tide._b.append(0, [1]), lambda: tide._b.attend(0, 0, rows, None, x, "a", x, None, 0)):
        with pytest.raises(TypeError):
            bad()
