"""The attention kernels run persistent thread blocks that take over item after item: batches of several hundred short
items (every block walks many, of one tile and of several, with one row tile and with two), items cut along the keys,
both head sizes, and launch shapes fixed larger than the batch.  Every output element and every LSE is compared with
the float64 oracle."""
import math

import numpy as np
import pytest

from oracle import cbuild
from oracle.paged_kv import PagedKVOracle
from paper_2608_10402_b200 import inputs
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("geom,n_rows,fixed", [((28, 4, 128, 16), 90, False), ((28, 4, 128, 32), 40, True), ((8, 2, 64, 16), 200, False),
                                               ((16, 1, 64, 32), 230, True), ((12, 4, 64, 16), 6, False)])
def test_many_short_items_per_thread_block(geom, n_rows, fixed):
    import torch
    from paper_2608_10402_b200 import tide
    HQ, HKV, D, S = geom
    G = HQ // HKV
    rng = np.random.default_rng(HQ + D + S + n_rows)
    scale = 1.0 / math.sqrt(D)
    edges = [16 // G + 1, 128 // G, 128 // G + 1, 256 // G, 256 // G + 1]        # around one and two row tiles
    new = [max(1, edges[b % 5]) if b % 2 else int(rng.integers(16 // G + 1, 600 // G + 2)) for b in range(n_rows)]
    prefix = [int(rng.choice([0, 1, 127, 128, 129])) if b % 3 == 0 else int(rng.integers(0, 700)) for b in range(n_rows)]
    if n_rows < 16:
        prefix[0], prefix[1] = 6000, 9001                                       # few items: cut along the keys and merged
    pages = sum((p + n + S - 1) // S for p, n in zip(prefix, new)) + 4
    max_pages = max((p + n + S - 1) // S for p, n in zip(prefix, new)) + 1
    T = sum(new)
    order = rng.permutation(pages).astype(np.int32)
    kv = tide.TideKV(HQ, HKV, D, S, pages, n_rows, max_pages, n_rows, T, free_order=order)
    orc = PagedKVOracle(pages, S, HKV, D, n_rows, max_pages, free_order=order)
    ids = list(range(n_rows))
    for o in (kv, orc):
        for t in ids:
            o.alloc(t)
    ip = np.concatenate([[0], np.cumsum(prefix)]).astype(np.int32)
    pk, pv = inputs.normal_bf16(rng, (int(ip[-1]), HKV, D)), inputs.normal_bf16(rng, (int(ip[-1]), HKV, D))
    kv.append(ids, ip, H.to_dev(pk, torch), H.to_dev(pv, torch))
    orc.append(ids, ip, pk, pv)
    ip = np.concatenate([[0], np.cumsum(new)]).astype(np.int32)
    nk, nv = inputs.normal_bf16(rng, (T, HKV, D)), inputs.normal_bf16(rng, (T, HKV, D))
    q = inputs.normal_bf16(rng, (T, HQ, D))
    rows = [(t, n, p + n) for t, (p, n) in enumerate(zip(prefix, new))]
    # results start 16 bytes behind a 32-byte boundary: the smallest alignment the call takes
    out = torch.zeros(T * HQ * D + 8, dtype=torch.int16, device="cuda")[8:].view(T, HQ, D)
    lse = torch.zeros((T, HQ), dtype=torch.float32, device="cuda")
    if fixed:
        kv.step_fix_grids(max_umma_items=4000, max_tokens=T)
        kv.step_begin(rows)
        kv.step_layer(0, H.to_dev(nk, torch), H.to_dev(nv, torch), H.to_dev(q, torch), scale, out, lse)
    else:
        kv.append(ids, ip, H.to_dev(nk, torch), H.to_dev(nv, torch))
        kv.attend(rows, H.to_dev(q, torch), scale, out, lse)
    assert kv.status() == tide.OK
    plan = kv.last_plan()
    assert plan["prefill_items"] > (0 if n_rows < 16 else 200) and plan["decode_items"] == 0
    assert (plan["merge_rows"] > 0) == (n_rows < 16)
    orc.append(ids, ip, nk, nv)
    ref_o, ref_l = cbuild.attend_paged(orc, rows, q, scale)
    H.check_outputs(H.from_dev(out), lse.cpu().numpy(), ref_o, ref_l, f"{geom}")
    kv.close()


@pytest.mark.parametrize("geom,n_rows,fixed", [((28, 4, 128, 16), 100, False), ((28, 4, 128, 32), 180, False), ((8, 2, 64, 16), 300, True),
                                               ((16, 1, 64, 32), 400, False), ((6, 2, 128, 16), 3, False), ((32, 8, 128, 16), 90, True)])
def test_many_decode_items_per_thread_block(geom, n_rows, fixed):
    """Decode-style rows from one key to several thousand, of one token or as many as still make one item: rows of one
    split beside rows whose splits are finished by different blocks, descriptors in the launch and uploaded."""
    import torch
    from paper_2608_10402_b200 import tide
    HQ, HKV, D, S = geom
    G = HQ // HKV
    rng = np.random.default_rng(HQ + 3 * D + S + n_rows)
    scale = 1.0 / math.sqrt(D)
    new = [int(rng.integers(1, 16 // G + 1)) for _ in range(n_rows)]
    edges = [0, 1, 63, 64, 65, 127, 128, 129, 511, 512]
    prefix = [edges[b % 10] if b % 2 else int(rng.integers(0, 900)) for b in range(n_rows)]
    for b in range(0, n_rows, 7):
        prefix[b] = int(rng.integers(2000, 9000))
    pages = sum((p + n + S - 1) // S for p, n in zip(prefix, new)) + 4
    max_pages = max((p + n + S - 1) // S for p, n in zip(prefix, new)) + 1
    T = sum(new)
    order = rng.permutation(pages).astype(np.int32)
    kv = tide.TideKV(HQ, HKV, D, S, pages, n_rows, max_pages, n_rows, T, free_order=order)
    orc = PagedKVOracle(pages, S, HKV, D, n_rows, max_pages, free_order=order)
    ids = list(range(n_rows))
    for o in (kv, orc):
        for t in ids:
            o.alloc(t)
    ip = np.concatenate([[0], np.cumsum(prefix)]).astype(np.int32)
    pk, pv = inputs.normal_bf16(rng, (int(ip[-1]), HKV, D)), inputs.normal_bf16(rng, (int(ip[-1]), HKV, D))
    kv.append(ids, ip, H.to_dev(pk, torch), H.to_dev(pv, torch))
    orc.append(ids, ip, pk, pv)
    ip = np.concatenate([[0], np.cumsum(new)]).astype(np.int32)
    nk, nv = inputs.normal_bf16(rng, (T, HKV, D)), inputs.normal_bf16(rng, (T, HKV, D))
    q = inputs.normal_bf16(rng, (T, HQ, D))
    rows = [(t, n, p + n) for t, (p, n) in enumerate(zip(prefix, new))]
    out = torch.zeros((T, HQ, D), dtype=torch.int16, device="cuda")
    lse = torch.zeros((T, HQ), dtype=torch.float32, device="cuda")
    dq = H.to_dev(q, torch)
    if fixed:
        kv.step_fix_grids(max_decode_items=3000, max_tokens=T)
        kv.step_begin(rows)
        kv.step_layer(0, H.to_dev(nk, torch), H.to_dev(nv, torch), dq, scale, out, lse)
    else:
        kv.append(ids, ip, H.to_dev(nk, torch), H.to_dev(nv, torch))
        kv.attend(rows, dq, scale, out, lse)
    assert kv.status() == tide.OK
    plan = kv.last_plan()
    assert plan["prefill_items"] == 0 and plan["merge_rows"] > 0 and (n_rows < 10 or plan["decode_items"] > 296)
    orc.append(ids, ip, nk, nv)
    ref_o, ref_l = cbuild.attend_paged(orc, rows, q, scale)
    H.check_outputs(H.from_dev(out), lse.cpu().numpy(), ref_o, ref_l, f"{geom}")
    # a second call finds the finished-split counters at zero again and gives the same bits
    first = out.clone()
    out.zero_()
    kv.attend(rows, dq, scale, out, lse)
    assert kv.status() == tide.OK and torch.equal(first, out)
    kv.close()


@pytest.mark.parametrize("geom,lens,cut", [((28, 4, 128, 16), [(0, 300)], False), ((28, 4, 128, 16), [(1500, 17)], True),
                                           ((6, 2, 128, 16), [(1280, 6), (2570, 300), (1, 90)], True), ((12, 4, 64, 16), [(0, 900), (2305, 31)], True),
                                           ((8, 1, 128, 32), [(383, 20), (9001, 3), (40, 2), (767, 64)], True),
                                           ((28, 4, 128, 16), [(6000 + 7 * i, 2 if i % 2 else 20 + i) for i in range(4)], True),
                                           ((28, 4, 128, 16), [(900 + 7 * i, 20 + i) for i in range(19)], False)])
def test_few_resume_rows_cut_along_their_keys(geom, lens, cut):
    """Resume rows whose items are few are cut along the keys where that is worth a merge: pieces that begin behind the last
    key of a row tile's tokens, rows shorter than a piece beside split ones, decode rows beside them."""
    import torch
    from paper_2608_10402_b200 import tide
    HQ, HKV, D, S = geom
    rng = np.random.default_rng(HQ + D + S + len(lens))
    scale = 1.0 / math.sqrt(D)
    lens = [(p, n if n == 2 and HQ // HKV <= 8 else max(n, 16 // (HQ // HKV) + 1)) for p, n in lens]
    n_rows, T = len(lens), sum(n for _, n in lens)
    max_pages = max((p + n + S - 1) // S for p, n in lens) + 1
    pages = n_rows * max_pages
    order = rng.permutation(pages).astype(np.int32)
    kv = tide.TideKV(HQ, HKV, D, S, pages, n_rows, max_pages, n_rows, T, free_order=order)
    orc = PagedKVOracle(pages, S, HKV, D, n_rows, max_pages, free_order=order)
    ids = list(range(n_rows))
    for o in (kv, orc):
        for t in ids:
            o.alloc(t)
    for part in (0, 1):
        ip = np.concatenate([[0], np.cumsum([x[part] for x in lens])]).astype(np.int32)
        nk, nv = inputs.normal_bf16(rng, (int(ip[-1]), HKV, D)), inputs.normal_bf16(rng, (int(ip[-1]), HKV, D))
        if ip[-1]:
            kv.append(ids, ip, H.to_dev(nk, torch), H.to_dev(nv, torch))
            orc.append(ids, ip, nk, nv)
    q = inputs.normal_bf16(rng, (T, HQ, D))
    rows = [(t, n, p + n) for t, (p, n) in enumerate(lens)]
    out = torch.zeros((T, HQ, D), dtype=torch.int16, device="cuda")
    lse = torch.zeros((T, HQ), dtype=torch.float32, device="cuda")
    kv.attend(rows, H.to_dev(q, torch), scale, out, lse)
    assert kv.status() == tide.OK
    plan = kv.last_plan()
    whole = sum(HKV * -(-n * (HQ // HKV) // 256) for _, n in lens if n * (HQ // HKV) > 16)
    if cut:
        assert plan["prefill_items"] > whole and plan["merge_rows"] > 0
    else:
        assert plan["prefill_items"] == whole
    ref_o, ref_l = cbuild.attend_paged(orc, rows, q, scale)
    H.check_outputs(H.from_dev(out), lse.cpu().numpy(), ref_o, ref_l, f"{geom}")
    kv.close()


@pytest.mark.parametrize("geom,ctx,pieces", [((28, 4, 128, 16), [1024], [4]), ((28, 4, 128, 16), [16000], [32]), ((28, 4, 128, 32), [4000] * 4, [8] * 4),
                                             ((16, 1, 128, 16), [40001, 130], [40, 1]), ((12, 4, 64, 16), [9000, 2047, 1], [24, 6, 1]),
                                             ((6, 2, 128, 16), [70000], [69]),
                                             ((28, 4, 128, 16), [250 + 250 * i for i in range(16)], [1, 1] + [2 + i // 2 for i in range(14)])])
def test_few_decode_rows_and_their_merge(geom, ctx, pieces):
    """Decode rows that are cut for the merge of their pieces: up to eight pieces, whole and ragged batches of eight, more
    than thirty-two; one block per SM and two."""
    import torch
    from paper_2608_10402_b200 import tide
    HQ, HKV, D, S = geom
    rng = np.random.default_rng(HQ + D + len(ctx) + ctx[0])
    scale, n = 1.0 / math.sqrt(D), len(ctx)
    max_pages = (max(ctx) + S) // S + 1
    pages = sum((c + S) // S + 1 for c in ctx)
    order = rng.permutation(pages).astype(np.int32)
    kv = tide.TideKV(HQ, HKV, D, S, pages, n, max_pages, n, max(ctx), free_order=order)
    orc = PagedKVOracle(pages, S, HKV, D, n, max_pages, free_order=order)
    for t, c in enumerate(ctx):
        nk, nv = inputs.normal_bf16(rng, (c, HKV, D)), inputs.normal_bf16(rng, (c, HKV, D))
        for o, k, v in ((kv, H.to_dev(nk, torch), H.to_dev(nv, torch)), (orc, nk, nv)):
            o.alloc(t)
            o.append([t], [0, c], k, v)
    q = inputs.normal_bf16(rng, (n, HQ, D))
    rows = [(t, 1, c) for t, c in enumerate(ctx)]
    out = torch.zeros((n, HQ, D), dtype=torch.int16, device="cuda")
    lse = torch.zeros((n, HQ), dtype=torch.float32, device="cuda")
    kv.attend(rows, H.to_dev(q, torch), scale, out, lse)
    assert kv.status() == tide.OK
    plan = kv.last_plan()
    assert plan["decode_items"] == HKV * sum(pieces) and plan["merge_rows"] == HQ * sum(p > 1 for p in pieces)
    ref_o, ref_l = cbuild.attend_paged(orc, rows, q, scale)
    H.check_outputs(H.from_dev(out), lse.cpu().numpy(), ref_o, ref_l, f"{geom}")
    kv.close()


@pytest.mark.parametrize("geom", [(28, 4, 128, 16), (12, 4, 64, 16)])
@pytest.mark.parametrize("layers", [1, 2])
def test_steps_queued_without_waiting_follow_one_another(geom, layers):
    """Kernels of one stream overlap at their edges: steps queued back to back (decode rows, resume rows and split rows
    in one batch; their own output buffers) each see the tokens of the steps before them and nothing of those after."""
    import torch
    from paper_2608_10402_b200 import tide
    from oracle.layers import LayeredKVOracle
    HQ, HKV, D, S = geom
    rng = np.random.default_rng(HQ + D + layers)
    scale = 1.0 / math.sqrt(D)
    B, steps = 9, 12
    prefix = [0, 15, 16, 130, 700, 1500, 2500, 60, 300]
    cnt = [[1 if (b + s) % 3 else int(rng.integers(1, 70)) for b in range(B)] for s in range(steps)]
    pages = sum((p + sum(c[b] for c in cnt) + S - 1) // S for b, p in enumerate(prefix)) + 4
    T = max(sum(c) for c in cnt)
    kv = tide.TideKV(HQ, HKV, D, S, pages, B, pages, B, max(T, 128), num_layers=layers)
    orc = LayeredKVOracle(layers, num_pages=pages, page_size=S, num_kv_heads=HKV, head_dim=D, max_tasks=B, max_pages_per_task=pages)
    ids = list(range(B))
    queue = []
    for s in range(-1, steps):
        n = prefix if s < 0 else cnt[s]
        ip = np.concatenate([[0], np.cumsum(n)]).astype(np.int32)
        shape = lambda h: (layers, int(ip[-1]), h, D)
        k, v, q = (inputs.normal_bf16(rng, shape(h)) for h in (HKV, HKV, HQ))
        queue.append((ip, k, v, q, *(H.to_dev(x, torch) for x in (k, v, q)), torch.zeros(shape(HQ), dtype=torch.int16, device="cuda"),
                      torch.zeros(shape(HQ)[:3], dtype=torch.float32, device="cuda")))
    for t in ids:
        kv.alloc(t)
        orc.alloc(t)
    ip, _, _, _, dk, dv, *_ = queue[0]
    kv.extend(ids, ip)
    for l in range(layers):
        kv.write(l, ids, ip, dk[l], dv[l])
    torch.cuda.synchronize()
    length = list(prefix)
    for ip, _, _, _, dk, dv, dq, out, lse in queue[1:]:
        length = [a + int(b) for a, b in zip(length, np.diff(ip))]
        rows = [(t, int(ip[t + 1] - ip[t]), length[t]) for t in ids]
        if layers > 1:
            kv.step_begin(rows)
            for l in range(layers):
                kv.step_layer(l, dk[l], dv[l], dq[l], scale, out[l], lse[l])
        else:
            kv.append(ids, ip, dk[0], dv[0])
            kv.attend(rows, dq[0], scale, out[0], lse[0])
    assert kv.status() == tide.OK
    orc.append(ids, *queue[0][:3])
    for s, (ip, k, v, q, _, _, _, out, lse) in enumerate(queue[1:]):
        orc.append(ids, ip, k, v)
        rows = [(t, int(ip[t + 1] - ip[t]), orc.task_len(t)) for t in ids]
        for l in range(layers):
            ref_o, ref_l = cbuild.attend_paged(orc.layer(l), rows, q[l], scale)
            H.check_outputs(H.from_dev(out[l]), lse[l].cpu().numpy(), ref_o, ref_l, f"step {s}, layer {l}")
    kv.close()


@pytest.mark.parametrize("geom", [(16, 16, 128, 16), (16, 16, 128, 32), (32, 16, 64, 16), (16, 16, 64, 32)])
def test_ragged_ends_leave_the_next_item_alone(geom):
    """Every item ends inside a 16-key block, whose unused V slots its consumers clear; the stage is filled again at once
    for the block's next item.  Few keys and large values: a slot lost to the item before shows far above the tolerance."""
    import torch
    from paper_2608_10402_b200 import tide
    HQ, HKV, D, S = geom
    rng = np.random.default_rng(HQ + D + S)
    scale, n = 1.0 / math.sqrt(D), 120
    ctx = [16 * int(rng.integers(0, 13)) + int(rng.integers(1, 16)) for _ in range(n)]
    pages, max_pages = sum((c + S - 1) // S for c in ctx) + 1, 208 // S + 1
    order = rng.permutation(pages).astype(np.int32)
    kv = tide.TideKV(HQ, HKV, D, S, pages, n, max_pages, n, sum(ctx), free_order=order)
    orc = PagedKVOracle(pages, S, HKV, D, n, max_pages, free_order=order)
    ip = np.concatenate([[0], np.cumsum(ctx)]).astype(np.int32)
    k = inputs.normal_bf16(rng, (int(ip[-1]), HKV, D))
    v = inputs.f32_to_bf16_bits(8.0 + 8.0 * rng.random((int(ip[-1]), HKV, D)).astype(np.float32))
    for o in (kv, orc):
        for t in range(n):
            o.alloc(t)
    kv.append(list(range(n)), ip, H.to_dev(k, torch), H.to_dev(v, torch))
    orc.append(list(range(n)), ip, k, v)
    q = inputs.normal_bf16(rng, (n, HQ, D))
    dq, rows = H.to_dev(q, torch), [(t, 1, c) for t, c in enumerate(ctx)]
    outs = [torch.zeros((n, HQ, D), dtype=torch.int16, device="cuda") for _ in range(20)]
    lse = torch.zeros((n, HQ), dtype=torch.float32, device="cuda")
    for out in outs:
        kv.attend(rows, dq, scale, out, lse)
    assert kv.status() == tide.OK and kv.last_plan()["decode_items"] == n * HKV
    ref_o, ref_l = cbuild.attend_paged(orc, rows, q, scale)
    H.check_outputs(H.from_dev(outs[0]), lse.cpu().numpy(), ref_o, ref_l, f"{geom}")
    assert all(torch.equal(outs[0], o) for o in outs[1:])
    kv.close()
