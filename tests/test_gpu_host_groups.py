"""Host-buffer steps cut into groups of tokens: rows longer than a group are cut too, groups run on two streams with
halves of the partials, and two steps follow one another on the same tasks.  Page tables and cache bits are compared with
the oracle exactly, outputs within the tolerance."""
import math

import numpy as np
import pytest

from oracle import cbuild
from oracle.paged_kv import PagedKVOracle
from paper_2608_10402_b200 import inputs
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("geom", [(28, 4, 128, 16), (16, 1, 64, 32)])
@pytest.mark.parametrize("groups", [1, 2, 4, 7])
def test_rows_are_cut_between_groups(geom, groups):
    import torch
    from paper_2608_10402_b200 import tide
    HQ, HKV, D, S = geom
    rng = np.random.default_rng(HQ + D + groups)
    scale = 1.0 / math.sqrt(D)
    prefix = [0, 700, 15, 2500, 3000, 1, 64, 900]
    steps = [[700, 1, 1, 1, 333, 1, 160, 17], [1, 1, 2, 1, 1, 900, 1, 1]]
    n = len(prefix)
    pages = sum((p + sum(s[b] for s in steps) + S - 1) // S for b, p in enumerate(prefix)) + 4
    order = rng.permutation(pages).astype(np.int32)
    kv = tide.TideKV(HQ, HKV, D, S, pages, n, pages, n, max(map(sum, steps)), free_order=order)
    kv.tune(tide.TUNE_HOST_STEP_CHUNKS, groups)
    kv.tune(tide.TUNE_HOST_ZERO_COPY, 0)
    orc = PagedKVOracle(pages, S, HKV, D, n, pages, free_order=order)
    ids = list(range(n))
    for o in (kv, orc):
        for t in ids:
            o.alloc(t)
    ip = np.concatenate([[0], np.cumsum(prefix)]).astype(np.int32)
    k, v = (inputs.normal_bf16(rng, (int(ip[-1]), HKV, D)) for _ in range(2))
    kv.append(ids, ip, H.to_dev(k, torch), H.to_dev(v, torch))
    orc.append(ids, ip, k, v)
    pin = lambda a: torch.from_numpy(np.ascontiguousarray(a).view(np.int16)).pin_memory()
    for cnt in steps:
        T = sum(cnt)
        ip = np.concatenate([[0], np.cumsum(cnt)]).astype(np.int32)
        k, v, q = (inputs.normal_bf16(rng, (T, h, D)) for h in (HKV, HKV, HQ))
        out = torch.zeros((T, HQ, D), dtype=torch.int16).pin_memory()
        lse = torch.zeros((T, HQ), dtype=torch.float32).pin_memory()
        orc.append(ids, ip, k, v)
        rows = [(t, c, orc.task_len(t)) for t, c in zip(ids, cnt)]
        kv.step_host(rows, pin(k), pin(v), pin(q), scale, out, lse)
        assert kv.status() == tide.OK and kv.usage() == (orc.used_tokens(), orc.free_pages())
        ref_o, ref_l = cbuild.attend_paged(orc, rows, q, scale)
        H.check_outputs(out.numpy().view(np.uint16), lse.numpy(), ref_o, ref_l, f"{cnt}")
        for t in ids:
            assert np.array_equal(kv.page_table(t), orc.page_table(t))
            gk, gv = kv.read(t)
            ok, ov = orc.read(t)
            assert np.array_equal(H.from_dev(gk), ok) and np.array_equal(H.from_dev(gv), ov)
    kv.close()
