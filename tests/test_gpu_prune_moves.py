"""Pruning moves a task's tail inside its own pages: shifts from one token to more than the tail (both kernels and the
line between them), tails around the runs and chains they work in, both head sizes and page sizes, several layers, and
several tasks in a row without waiting.  Cache bits and page tables are compared with the oracle exactly."""
import numpy as np
import pytest

from oracle.layers import LayeredKVOracle
from paper_2608_10402_b200 import inputs
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("geom,layers", [((28, 4, 128, 16), 1), ((6, 3, 64, 16), 2), ((8, 1, 128, 32), 1), ((8, 2, 64, 32), 1)])
def test_tails_move_in_place(geom, layers):
    import torch
    from paper_2608_10402_b200 import tide
    HQ, HKV, D, S = geom
    rng = np.random.default_rng(HQ + HKV + D + S)
    # (kept prefix, shift, tail)
    shapes = [(0, 1, 700), (5, 2, 1), (16, 16, 1025), (17, 63, 600), (17, 64, 600), (3, 65, 64), (31, 128, 1100), (100, 257, 256),
              (1, 400, 3000), (40, 900, 10), (7, 15, 0), (0, 64, 513), (33, 3, 512), (33, 31, 511)]
    n = len(shapes)
    length = [sum(x) for x in shapes]
    pages = sum((l + S - 1) // S for l in length) + 8
    order = rng.permutation(pages).astype(np.int32)
    kv = tide.TideKV(HQ, HKV, D, S, pages, n, pages, n, 256, free_order=order, num_layers=layers)
    orc = LayeredKVOracle(layers, num_pages=pages, page_size=S, num_kv_heads=HKV, head_dim=D, max_tasks=n, max_pages_per_task=pages,
                          free_order=order)
    ip = np.concatenate([[0], np.cumsum(length)]).astype(np.int32)
    k, v = (inputs.normal_bf16(rng, (layers, int(ip[-1]), HKV, D)) for _ in range(2))
    ids = list(range(n))
    for o in (kv, orc):
        for t in ids:
            o.alloc(t)
    kv.extend(ids, ip)
    for l in range(layers):
        kv.write(l, ids, ip, H.to_dev(k[l], torch), H.to_dev(v[l], torch))
    orc.append(ids, ip, k, v)

    def same():
        assert kv.status() == tide.OK and kv.usage() == (orc.used_tokens(), orc.free_pages())
        for t in ids:
            assert np.array_equal(kv.page_table(t), orc.page_table(t))
            for l in range(layers):
                gk, gv = kv.read(t, layer=l)
                ok, ov = orc.read(l, t)
                assert np.array_equal(H.from_dev(gk), ok) and np.array_equal(H.from_dev(gv), ov), (t, shapes[t], l)

    for t, (keep, shift, _) in enumerate(shapes):        # one behind the other: moves of different tasks overlap
        kv.prune(t, keep, keep + shift)
        orc.prune(t, keep, keep + shift)
    same()
    for t in ids * 2:                                    # the same task again directly behind its own move
        m = kv.task_len(t)
        if m > 40:
            for o in (kv, orc):
                o.prune(t, 3, 3 + m // 9)
                o.prune(t, 1, 2)
    # tokens appended into the freed pages directly behind the moves
    ip = np.arange(n + 1, dtype=np.int32) * 9
    k, v = (inputs.normal_bf16(rng, (layers, 9 * n, HKV, D)) for _ in range(2))
    kv.extend(ids, ip)
    for l in range(layers):
        kv.write(l, ids, ip, H.to_dev(k[l], torch), H.to_dev(v[l], torch))
    orc.append(ids, ip, k, v)
    same()
    kv.close()


@pytest.mark.parametrize("geom,layers", [((28, 4, 128, 16), 1), ((8, 2, 64, 32), 2)])
def test_chains_cut_into_segments(geom, layers):
    """Chains of as many links as a segment holds, one more and one less, and of 32 segments'; the longest of a shift of two; fewer
    chains than a block holds, and a last block that is not full; tails that fill the chip with fewer segments."""
    import torch
    from paper_2608_10402_b200 import tide
    HQ, HKV, D, S = geom
    rng = np.random.default_rng(7 * HQ + D)
    shapes = [(3, 40, 40 * 5), (3, 40, 40 * 5 + 1), (0, 7, 7 * 6 - 1), (1, 2, 2 * 160), (1, 2, 2 * 160 + 1), (15, 33, 33 * 32 + 5), (2, 2, 8192), (2, 2, 8193),
              (5, 600, 4000), (0, 31, 1), (9, 1000, 6000), (100, 65, 64 * 65),
              # last cuts taken back; a shift of two by runs
              (3, 64, 64 * 300 + 5), (7, 32, 32 * 520 + 1), (2, 2, 2 * 8192 + 1)]
    length = [sum(x) for x in shapes]
    n, pages = len(shapes), sum((l + S - 1) // S for l in length) + 4
    order = rng.permutation(pages).astype(np.int32)
    kv = tide.TideKV(HQ, HKV, D, S, pages, n, pages, n, 256, free_order=order, num_layers=layers)
    orc = LayeredKVOracle(layers, num_pages=pages, page_size=S, num_kv_heads=HKV, head_dim=D, max_tasks=n, max_pages_per_task=pages, free_order=order)
    ids, ip = list(range(n)), np.concatenate([[0], np.cumsum(length)]).astype(np.int32)
    k, v = (inputs.normal_bf16(rng, (layers, int(ip[-1]), HKV, D)) for _ in range(2))
    for o in (kv, orc):
        for t in ids:
            o.alloc(t)
    kv.extend(ids, ip)
    for l in range(layers):
        kv.write(l, ids, ip, H.to_dev(k[l], torch), H.to_dev(v[l], torch))
    orc.append(ids, ip, k, v)
    for t, (keep, shift, _) in enumerate(shapes):
        kv.prune(t, keep, keep + shift)
        orc.prune(t, keep, keep + shift)
    for t in ids:
        for l in range(layers):
            (gk, gv), (ok, ov) = kv.read(t, layer=l), orc.read(l, t)
            assert np.array_equal(H.from_dev(gk), ok) and np.array_equal(H.from_dev(gv), ov), (shapes[t], l)
    kv.close()
