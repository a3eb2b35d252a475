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


def test_rows_are_records_or_triples_of_int32(tide):
    x = np.zeros(4)
    call = lambda rows: (tide._b.attend(0, 0, rows, None, x, 0.5, x, None, 0), tide._b.step_begin(0, rows, 0),
                         tide._b.step_host(0, rows, x, x, x, 0.5, x, None, 0))
    record = np.dtype([("task", np.int32), ("q_len", np.int32), ("ctx_len", np.int32)])
    for good in (tide.rows_array([(0, 1, 5), (1, 2, 7)]), tide.rows_array([]), np.zeros((5, 3), np.int32), np.zeros((0, 3), np.int32), np.zeros(5, record)):
        assert call(good) == (tide.ERR_INVALID_ARG,) * 3
    for bad in (np.zeros((5, 3), np.int64), np.zeros((5, 3), np.float32), np.zeros((5, 3), np.uint32), np.zeros((5, 3), ">i4"), np.zeros(15, np.int32),
                np.zeros((3, 5), np.int32), np.zeros((5, 4), np.int32), np.zeros((4, 2, 3), np.int32), bytes(24), bytearray(7), np.zeros(5, "V12"),
                np.zeros(5, [("a", np.int32), ("b", np.float32), ("c", np.int32)]), (tide.ctypes.c_int32 * 6)()):
        for f in (lambda: tide._b.attend(0, 0, bad, None, x, 0.5, x, None, 0), lambda: tide._b.step_begin(0, bad, 0),
                  lambda: tide._b.step_host(0, bad, x, x, x, 0.5, x, None, 0)):
            with pytest.raises(TypeError):
                f()


def test_pointers_are_numbers_arrays_and_tensors(tide):
    """numpy arrays by the address of their first element, whatever their strides and type; nothing else that happens to
    export a buffer - a numpy integer that holds an address is not the address of that integer."""
    import torch
    rows = tide.rows_array([(0, 1, 5)])
    call = lambda p: tide._b.attend(0, 0, rows, None, p, 0.5, p, p, 0)
    a = np.zeros((4, 4))
    for good in (None, 4096, a, a[:, :2], a[::-1], a.T, np.zeros(()), np.zeros(0), np.zeros(3, "M8[s]"), np.frombuffer(b"1234", np.int32),
                 torch.zeros(3), torch.zeros((3, 3), dtype=torch.bfloat16).t()):
        assert call(good) == tide.ERR_INVALID_ARG
    for bad in (np.int64(4096), b"1234", bytearray(4), memoryview(b"1234"), (tide.ctypes.c_int32 * 6)(), tide.ctypes.c_void_p(4096), 4096.0, "a"):
        with pytest.raises((TypeError, AttributeError)):
            call(bad)
