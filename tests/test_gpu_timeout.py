"""The bounded waits inside the attention kernels, made to run out WITHOUT any fault: a test hook lets the K/V
producer of one work item leave out the first stage, so the consumers' wait for it reaches its (shortened) time
limit.  The kernel must return by itself, tide_status must report the time-out exactly once, and the same handle
must then compute correct attention again."""
import math
import time

import numpy as np
import pytest

from oracle import cbuild
from oracle.paged_kv import PagedKVOracle
from paper_2608_10402_b200 import inputs
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,geom,p,n", [("warp-MMA decode kernel", (8, 2, 64, 16), 300, 1),
                                           ("warp-MMA decode kernel, head size 128", (28, 4, 128, 16), 700, 1),
                                           ("warp-MMA tile kernel", (8, 2, 64, 16), 150, 40),
                                           ("tcgen05 kernel, head size 64", (8, 2, 64, 16), 150, 40),
                                           ("tcgen05 kernel", (28, 4, 128, 16), 200, 40)])
def test_a_wait_that_runs_out_is_reported_once_and_the_handle_stays_usable(kind, geom, p, n):
    import torch
    from paper_2608_10402_b200 import tide
    HQ, HKV, D, S = geom
    rng = np.random.default_rng(p + n)
    L = p + n
    pages = (L + S - 1) // S + 2
    kv = tide.TideKV(HQ, HKV, D, S, pages, 2, pages, 2, max(n, 4))
    if kind == "warp-MMA tile kernel":
        kv.tune(tide.TUNE_UMMA_TILE_KEYS, 64)                 # the tcgen05 kernel with these takes no 64-wide heads
    orc = PagedKVOracle(pages, S, HKV, D, 2, pages)
    k, v = inputs.normal_bf16(rng, (L, HKV, D)), inputs.normal_bf16(rng, (L, HKV, D))
    for o in (kv, orc):
        o.alloc(0)
    kv.append([0], [0, L], H.to_dev(k, torch), H.to_dev(v, torch))
    orc.append([0], [0, L], k, v)
    rows = [(0, n, L)]
    q = inputs.normal_bf16(rng, (n, HQ, D))
    scale = 1.0 / math.sqrt(D)
    out = torch.zeros((n, HQ, D), dtype=torch.int16, device="cuda")
    lse = torch.zeros((n, HQ), dtype=torch.float32, device="cuda")
    assert kv.status() == tide.OK

    kv.tune(tide.TUNE_WAIT_LIMIT_US, 2000)                    # 2 ms instead of 2 s
    kv.tune(tide.TUNE_DROP_FIRST_STAGE, 1)                    # armed for the next attention call only
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    kv.attend(rows, H.to_dev(q, torch), scale, out, lse)      # the call itself is asynchronous and succeeds
    st = kv.status()                                          # synchronises: the kernel came back by itself
    elapsed = time.perf_counter() - t0
    assert st == tide.ERR_DEVICE_TIMEOUT, f"{kind}: status {st}"
    assert elapsed < 2.0, f"{kind}: {elapsed:.3f} s for waits bounded at 2 ms"
    assert (kv.last_plan()["prefill_items"] == HKV * -(-n * (HQ // HKV) // (64 if "tile" in kind else 256))) == (n > 1)
    assert kv.status() == tide.OK                             # reported once, then cleared

    kv.tune(tide.TUNE_WAIT_LIMIT_US, 2_000_000)
    out.zero_()
    lse.zero_()
    kv.attend(rows, H.to_dev(q, torch), scale, out, lse)      # the hook is spent: this is an ordinary call
    assert kv.status() == tide.OK
    ref_o, ref_l = cbuild.attend_paged(orc, rows, q, scale)
    H.check_outputs(H.from_dev(out), lse.cpu().numpy(), ref_o, ref_l, kind + " after the time-out")
    gk, gv = kv.read(0)
    assert np.array_equal(H.from_dev(gk), k) and np.array_equal(H.from_dev(gv), v)     # the cache was never touched
    kv.close()


@pytest.mark.parametrize("geom,n,p,times", [((28, 4, 128, 16), 1, 1500, 1), ((16, 16, 128, 16), 1, 40, 16), ((16, 16, 64, 32), 1, 40, 16),
                                            ((8, 2, 64, 32), 1, 3000, 4), ((28, 4, 128, 16), 20, 180, 1), ((28, 4, 128, 16), 20, 5000, 1),
                                            ((8, 2, 64, 16), 30, 200, 1)])
def test_the_limit_does_not_count_the_kernel_in_front(geom, n, p, times):
    """A move of some 0.5 ms on a few thread blocks runs in front; the attention kernel starts beside it on the other
    SMs, fills its ring - with one item, or with all the items it may publish - and holds its consumers up until the move
    is complete, several limits later."""
    import torch
    from paper_2608_10402_b200 import tide
    HQ, HKV, D, S = geom
    rng = np.random.default_rng(HQ + D + n + p)
    scale, L, long = 1.0 / math.sqrt(D), p + n, 120_000
    tasks = 9                                                 # task 0 is moved, eight rows are attended
    max_pages = (long + S - 1) // S + 1
    pages = max_pages + (tasks - 1) * ((L + S - 1) // S) + 1
    kv = tide.TideKV(HQ, HKV, D, S, pages, tasks, max_pages, 8 * times, 8 * n * times)
    orc = PagedKVOracle(pages, S, HKV, D, tasks, max_pages)
    kv.alloc(0)
    big = torch.zeros((long, HKV, D), dtype=torch.int16, device="cuda")
    kv.append([0], [0, long], big, big)
    for t in range(1, tasks):
        k, v = inputs.normal_bf16(rng, (L, HKV, D)), inputs.normal_bf16(rng, (L, HKV, D))
        for o, a, b in ((kv, H.to_dev(k, torch), H.to_dev(v, torch)), (orc, k, v)):
            o.alloc(t)
            o.append([t], [0, L], a, b)
    rows = [(t, n, L) for t in range(1, tasks)] * times
    q = inputs.normal_bf16(rng, (len(rows) * n, HQ, D))
    dq = H.to_dev(q, torch)
    out = torch.zeros((len(rows) * n, HQ, D), dtype=torch.int16, device="cuda")
    lse = torch.zeros((len(rows) * n, HQ), dtype=torch.float32, device="cuda")
    kv.attend(rows, dq, scale, out, lse)
    torch.cuda.synchronize()
    kv.tune(tide.TUNE_WAIT_LIMIT_US, 100)
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    ev[0].record()
    kv.prune(0, 0, 1)                                         # by one: a few blocks move it, whatever its length
    ev[1].record()
    kv.prune(0, 0, 1)                                         # a series of its own: an event has come between
    kv.attend(rows, dq, scale, out, lse)
    assert kv.status() == tide.OK
    assert ev[0].elapsed_time(ev[1]) > 0.2, "the case is meant to have a long launch in front"
    ref_o, ref_l = cbuild.attend_paged(orc, rows, q, scale)
    H.check_outputs(H.from_dev(out), lse.cpu().numpy(), ref_o, ref_l, f"{geom}")
    kv.close()


def test_the_limit_does_not_count_the_tensor_kernel_that_decode_rows_run_beside():
    """Members of a group merge with their shared range's partials, which the tcgen05 kernel in front writes among items of
    0.2 ms; the decode kernel's other warps wait meanwhile."""
    import torch
    from paper_2608_10402_b200 import tide
    HQ, HKV, D, S = 28, 4, 128, 16
    rng = np.random.default_rng(5)
    scale, ctx, new, n_long, shared, own, m = 1.0 / math.sqrt(D), 16000, 36, 40, 4096, 900, 200
    max_pages = ctx // S + 1
    pages = n_long * (ctx // S + 1) + shared // S + m * (own // S + 2) + 8
    n = n_long + m
    kv = tide.TideKV(HQ, HKV, D, S, pages, n, max_pages, n, n_long * new + m)
    kv.tune(tide.TUNE_MIN_SAVED_BYTES, 0)
    some = lambda t: torch.randn((t, HKV, D), device="cuda", dtype=torch.float32).to(torch.bfloat16)
    for t in range(n_long):
        kv.alloc(t)
        kv.append([t], [0, ctx], some(ctx), some(ctx))
    kv.alloc(n_long)
    kv.append([n_long], [0, shared], some(shared), some(shared))
    for t in range(n_long + 1, n):
        kv.fork(n_long, t)
    for t in range(n_long, n):
        kv.append([t], [0, own], some(own), some(own))
    rows = [(t, new, ctx) for t in range(n_long)] + [(t, 1, shared + own) for t in range(n_long, n)]
    T = n_long * new + m
    q = torch.randn((T, HQ, D), device="cuda", dtype=torch.float32).to(torch.bfloat16)
    got = []
    for limit in (2_000_000, 100):
        kv.tune(tide.TUNE_WAIT_LIMIT_US, limit)
        out = torch.zeros((T, HQ, D), dtype=torch.bfloat16, device="cuda")
        lse = torch.zeros((T, HQ), dtype=torch.float32, device="cuda")
        kv.attend(rows, q, scale, out, lse)
        assert kv.status() == tide.OK, limit
        assert kv.last_sharing()["groups"] > 0
        got.append((out, lse))
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
    kv.close()
