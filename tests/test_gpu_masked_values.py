"""A query's result does not depend on the values of tokens behind it, not even infinite ones, as far as they lie in pieces
of the row that the query sees nothing of: pieces without a visible key drop out of the merge."""
import math

import numpy as np
import pytest

from oracle import cbuild
from oracle.paged_kv import PagedKVOracle
from paper_2608_10402_b200 import inputs
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("geom,n", [((28, 4, 128, 16), 2), ((8, 2, 64, 32), 3), ((28, 4, 128, 16), 30), ((8, 2, 64, 16), 30)])
@pytest.mark.parametrize("front", [1024, 6144])
@pytest.mark.parametrize("bad", [0x7F80, 0xFF80, 0x7FC0])     # the two infinities and a NaN, as bf16 bits
def test_an_infinite_value_behind_a_query_in_a_piece_of_its_own(geom, n, front, bad):
    """A row of n tokens whose last n - 1 fill the row's last piece: its first query sees nothing of it."""
    import torch
    from paper_2608_10402_b200 import tide
    HQ, HKV, D, S = geom
    rng = np.random.default_rng(HQ + D + n)
    scale, L = 1.0 / math.sqrt(D), front + n - 1
    pages = L // S + 2
    kv = tide.TideKV(HQ, HKV, D, S, pages, 1, pages, 1, L)
    orc = PagedKVOracle(pages, S, HKV, D, 1, pages)
    k, v = inputs.normal_bf16(rng, (L, HKV, D)), inputs.normal_bf16(rng, (L, HKV, D))
    q = inputs.normal_bf16(rng, (n, HQ, D))
    kv.alloc(0)
    orc.alloc(0)
    orc.append([0], [0, L], k, v)
    poisoned = v.copy()
    poisoned[front:] = bad
    kv.append([0], [0, L], H.to_dev(k, torch), H.to_dev(poisoned, torch))
    out = torch.zeros((n, HQ, D), dtype=torch.int16, device="cuda")
    lse = torch.zeros((n, HQ), dtype=torch.float32, device="cuda")
    kv.attend([(0, n, L)], H.to_dev(q, torch), scale, out, lse)
    assert kv.status() == tide.OK
    plan = kv.last_plan()
    pieces = (plan["decode_items"] + plan["prefill_items"]) // HKV
    assert plan["merge_rows"] == n * HQ and front % ((pieces - 1) * 128) == 0, "the last piece is meant to begin at `front`"
    ref_o, ref_l = cbuild.attend_paged(orc, [(0, n, L)], q, scale)
    H.check_outputs(H.from_dev(out)[:1], lse.cpu().numpy()[:1], ref_o[:1], ref_l[:1], f"{geom}")
    kv.close()


@pytest.mark.parametrize("geom", [(28, 4, 128, 16), (8, 2, 64, 32)])
@pytest.mark.parametrize("ctx", [1000, 2048, 2300, 12000])
def test_an_infinite_value_that_is_visible_stays_infinite(geom, ctx):
    """Pieces of a row in full batches of eight and fewer: one infinite element of one key makes that element of the result
    infinite, for the query heads of its KV head, and changes nothing else."""
    import torch
    from paper_2608_10402_b200 import tide
    HQ, HKV, D, S = geom
    rng = np.random.default_rng(HQ + D + ctx)
    scale, G = 1.0 / math.sqrt(D), HQ // HKV
    pages = ctx // S + 2
    kv = tide.TideKV(HQ, HKV, D, S, pages, 1, pages, 1, ctx)
    orc = PagedKVOracle(pages, S, HKV, D, 1, pages)
    k, v = inputs.normal_bf16(rng, (ctx, HKV, D)), inputs.normal_bf16(rng, (ctx, HKV, D))
    k = inputs.f32_to_bf16_bits(inputs.bf16_bits_to_f32(k) * np.float32(0.25))       # no weight so small that it vanishes
    q = inputs.normal_bf16(rng, (1, HQ, D))
    kv.alloc(0)
    orc.alloc(0)
    orc.append([0], [0, ctx], k, v)
    marked = v.copy()
    marked[ctx // 3, 1, 5], marked[ctx - 1, 0, D - 1] = 0x7F80, 0xFF80
    kv.append([0], [0, ctx], H.to_dev(k, torch), H.to_dev(marked, torch))
    out = torch.zeros((1, HQ, D), dtype=torch.int16, device="cuda")
    lse = torch.zeros((1, HQ), dtype=torch.float32, device="cuda")
    kv.attend([(0, 1, ctx)], H.to_dev(q, torch), scale, out, lse)
    assert kv.status() == tide.OK and kv.last_plan()["merge_rows"] == HQ
    bits = H.from_dev(out)
    assert (bits[0, G:2 * G, 5] == 0x7F80).all() and (bits[0, :G, D - 1] == 0xFF80).all()
    ref_o, ref_l = cbuild.attend_paged(orc, [(0, 1, ctx)], q, scale)
    bits[0, G:2 * G, 5], bits[0, :G, D - 1] = 0, 0
    ref_o[0, G:2 * G, 5], ref_o[0, :G, D - 1] = 0, 0
    H.check_outputs(bits, lse.cpu().numpy(), ref_o, ref_l, f"{geom}")
    kv.close()
