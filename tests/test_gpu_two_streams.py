"""One handle used from two streams: appends of other tasks on one stream come between the append and the attention of a
task on the other, with no event between the two streams there.  Attention calls share the workspace, so these are ordered
by events.  Outputs and LSEs are compared with the float64 oracle, step by step."""
import math

import numpy as np
import pytest

from oracle import cbuild
from oracle.paged_kv import PagedKVOracle
from paper_2608_10402_b200 import inputs
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("geom", [(28, 4, 128, 16), (8, 2, 64, 32)])
@pytest.mark.parametrize("fresh", [1, 40, 300])
def test_appends_on_another_stream_between_append_and_attend(geom, fresh):
    import torch
    from paper_2608_10402_b200 import tide
    HQ, HKV, D, S = geom
    rng = np.random.default_rng(HQ + D + fresh)
    scale, steps = 1.0 / math.sqrt(D), 8
    prefix = [2000, 900, 1300, 15]
    per_step = [fresh, 3, 500, 1]
    n = len(prefix)
    pages = sum((p + steps * c + S - 1) // S for p, c in zip(prefix, per_step)) + 4
    order = rng.permutation(pages).astype(np.int32)
    kv = tide.TideKV(HQ, HKV, D, S, pages, n, pages, n, 4096, free_order=order)
    orc = PagedKVOracle(pages, S, HKV, D, n, pages, free_order=order)
    bits = lambda t, h: inputs.normal_bf16(rng, (t, h, D))
    for t, p in enumerate(prefix):
        k, v = bits(p, HKV), bits(p, HKV)
        for o in (kv, orc):
            o.alloc(t)
        kv.append([t], [0, p], H.to_dev(k, torch), H.to_dev(v, torch))
        orc.append([t], [0, p], k, v)
    work = [[(bits(c, HKV), bits(c, HKV), bits(c, HQ)) for c in per_step] for _ in range(steps)]
    dev = [[tuple(H.to_dev(x, torch) for x in w) for w in step] for step in work]
    outs = [[(torch.zeros((c, HQ, D), dtype=torch.int16, device="cuda"), torch.zeros((c, HQ), dtype=torch.float32, device="cuda"))
             for c in per_step] for _ in range(steps)]
    sa, sb = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    length = list(prefix)
    for s in range(steps):
        def append(t, stream):
            kv.append([t], [0, per_step[t]], dev[s][t][0], dev[s][t][1], stream=stream)
            length[t] += per_step[t]

        def attend(t, stream):
            kv.attend([(t, per_step[t], length[t])], dev[s][t][2], scale, *outs[s][t], stream=stream)
        append(0, sb)
        append(1, sa)
        append(2, sa)
        attend(0, sb)
        sa.wait_stream(sb)
        append(3, sa)
        attend(1, sa)
        attend(2, sa)
        attend(3, sa)
        sb.wait_stream(sa)
    torch.cuda.synchronize()
    assert kv.status() == tide.OK
    for s in range(steps):
        for t in range(n):
            orc.append([t], [0, per_step[t]], work[s][t][0], work[s][t][1])
            ref_o, ref_l = cbuild.attend_paged(orc, [(t, per_step[t], orc.task_len(t))], work[s][t][2], scale)
            H.check_outputs(H.from_dev(outs[s][t][0]), outs[s][t][1].cpu().numpy(), ref_o, ref_l, f"step {s}, task {t}")
    kv.close()
