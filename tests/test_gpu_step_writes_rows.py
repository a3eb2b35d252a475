"""Layers of a step whose rows are all decode-style: the attention launch writes the step's K/V
rows itself.  Rows of one to as many tokens as still make a decode item, new tokens across pages, stages and pieces, long rows
cut into pieces; three steps in a row; a writer between two layers; and a wait that runs out, after which the cache must hold
every layer's rows.  Cache bits are compared with the oracle exactly, results within its tolerance."""
import math

import numpy as np
import pytest

from oracle import cbuild
from oracle.layers import LayeredKVOracle
from paper_2608_10402_b200 import inputs
from tests import helpers as H

pytestmark = pytest.mark.gpu
LAYERS = 3


class Both:
    """The library and the oracle, filled alike."""

    def __init__(self, geom, prefix, room):
        import torch
        from paper_2608_10402_b200 import tide
        self.torch, self.tide, self.geom = torch, tide, geom
        HQ, HKV, D, S = geom
        self.rng = rng = np.random.default_rng(HQ + HKV + D + S)
        n = len(prefix)
        pages = sum((p + room + S - 1) // S for p in prefix) + 16
        most = max((p + room + S - 1) // S for p in prefix) + 1
        order = rng.permutation(pages).astype(np.int32)
        self.kv = tide.TideKV(HQ, HKV, D, S, pages, n + 4, most, n, 4096, free_order=order, num_layers=LAYERS)
        self.orc = LayeredKVOracle(LAYERS, num_pages=pages, page_size=S, num_kv_heads=HKV, head_dim=D, max_tasks=n, max_pages_per_task=most,
                                   free_order=order)
        self.ids = list(range(n))
        for o in (self.kv, self.orc):
            for t in self.ids:
                o.alloc(t)
        ip = np.concatenate([[0], np.cumsum(prefix)]).astype(np.int32)
        k, v = self.rows(int(ip[-1])), self.rows(int(ip[-1]))
        self.kv.extend(self.ids, ip)
        for l in range(LAYERS):
            self.kv.write(l, self.ids, ip, H.to_dev(k[l], torch), H.to_dev(v[l], torch))
        self.orc.append(self.ids, ip, k, v)

    def rows(self, tokens):
        return np.stack([inputs.normal_bf16(self.rng, (tokens, self.geom[1], self.geom[2])) for _ in range(LAYERS)])

    def step(self, new, between=None, check=True):
        HQ, HKV, D, S = self.geom
        torch, kv, orc = self.torch, self.kv, self.orc
        ip = np.concatenate([[0], np.cumsum(new)]).astype(np.int32)
        T = int(ip[-1])
        k, v = self.rows(T), self.rows(T)
        q = np.stack([inputs.normal_bf16(self.rng, (T, HQ, D)) for _ in range(LAYERS)])
        orc.append(self.ids, ip, k, v)
        rows = [(t, c, orc.task_len(t)) for t, c in zip(self.ids, new)]
        out = torch.zeros((LAYERS, T, HQ, D), dtype=torch.int16, device="cuda")
        lse = torch.zeros((LAYERS, T, HQ), dtype=torch.float32, device="cuda")
        dk, dv, dq = H.to_dev(k, torch), H.to_dev(v, torch), H.to_dev(q, torch)
        kv.step_begin(rows)
        launches = []
        for l in range(LAYERS):
            if between:
                between(l)
            kv.step_layer(l, dk[l], dv[l], dq[l], 1.0 / math.sqrt(D), out[l], lse[l])
            launches.append(kv.last_plan()["kernel_launches"])
        self.last = (rows, k, v, q, out, lse)
        if check:
            assert kv.status() == self.tide.OK
            for l in range(LAYERS):
                ref_o, ref_l = cbuild.attend_paged(orc.layer(l), rows, q[l], 1.0 / math.sqrt(D))
                H.check_outputs(H.from_dev(out[l]), lse[l].cpu().numpy(), ref_o, ref_l, f"layer {l}")
        return launches

    def same_bits(self):
        for l in range(LAYERS):
            for t in self.ids:
                gk, gv = self.kv.read(t, layer=l)
                ok, ov = self.orc.read(l, t)
                assert np.array_equal(H.from_dev(gk), ok) and np.array_equal(H.from_dev(gv), ov), (l, t)


@pytest.mark.parametrize("geom", [(28, 4, 128, 16), (8, 2, 64, 16), (12, 4, 64, 32), (16, 1, 128, 32), (6, 3, 64, 16), (3, 3, 128, 32), (2, 2, 64, 16)])
def test_rows_are_written_by_the_attention_launch(geom):
    G = geom[0] // geom[1]
    most = 16 // G
    prefix = [0, 1, 14, 15, 16, 31, 47, 62, 63, 64, 126, 127, 128, 129, 255, 511, 6000, 6143]
    b = Both(geom, prefix, 3 * most)
    for r in range(3):                                        # the last piece of a long row ends before, at or behind a boundary
        new = [1 if r == 0 else int(b.rng.integers(1, most + 1)) for _ in prefix]
        new[-1] = most if r else 1
        assert b.step(new) == [1, 1, 1]
    b.same_bits()
    b.kv.close()


def test_a_writer_between_two_layers_goes_in_front():
    b = Both((8, 2, 64, 16), [300, 40, 2000], 8)
    extra, torch = {}, b.torch

    def between(l):
        if l != 1:
            return
        # the last 20 rows of task 2 - 19 in front of the step's own, which its launch writes again - on every layer
        k, v = b.rows(20), b.rows(20)
        for x in range(LAYERS):
            b.kv.write(x, [2], [0, 20], H.to_dev(k[x], torch), H.to_dev(v[x], torch))
        extra["k"], extra["v"] = k, v

    assert b.step([1, 1, 1], between, check=False) == [1, 1, 1]
    assert b.kv.status() == b.tide.OK
    for l in range(LAYERS):
        gk, gv = (H.from_dev(x) for x in b.kv.read(2, layer=l))
        ok, _ = b.orc.read(l, 2)
        assert np.array_equal(gk[-20:-1], extra["k"][l][:19]) and np.array_equal(gv[-20:-1], extra["v"][l][:19])
        assert np.array_equal(gk[-1], ok[-1] if l else extra["k"][l][19]) and np.array_equal(gk[:-20], ok[:-20])
    # the layers behind the writer have seen its rows
    rows, k, v, q, out, lse = b.last
    b.orc.truncate(2, b.orc.task_len(2) - 20)
    b.orc.append([2], np.array([0, 20], np.int32), np.concatenate([extra["k"][:, :19], k[:, 2:]], axis=1), np.concatenate([extra["v"][:, :19], v[:, 2:]], axis=1))
    for l in (1, 2):
        ref_o, ref_l = cbuild.attend_paged(b.orc.layer(l), rows, q[l], 1.0 / math.sqrt(b.geom[2]))
        H.check_outputs(H.from_dev(out[l]), lse[l].cpu().numpy(), ref_o, ref_l, f"layer {l}")
    b.kv.close()


@pytest.mark.parametrize("geom", [(16, 16, 128, 16), (8, 2, 64, 32)])
@pytest.mark.parametrize("over", ["k", "v"])
def test_results_over_the_new_rows(geom, over):
    HQ, HKV, D, S = geom
    b = Both(geom, [40 + 37 * i for i in range(60)], 2)
    torch, n = b.torch, len(b.ids)
    k, v = b.rows(n), b.rows(n)
    q = np.stack([inputs.normal_bf16(b.rng, (n, HQ, D)) for _ in range(LAYERS)])
    b.orc.append(b.ids, np.arange(n + 1, dtype=np.int32), k, v)
    rows = [(t, 1, b.orc.task_len(t)) for t in b.ids]
    dk, dv, dq = H.to_dev(k, torch), H.to_dev(v, torch), H.to_dev(q, torch)
    b.kv.step_begin(rows)
    outs = []
    for l in range(LAYERS):
        # the rows lie where the results of the first heads go
        out = torch.zeros((n, HQ, D), dtype=torch.int16, device="cuda")
        new = out.view(-1)[:n * HKV * D].view(n, HKV, D)
        new.copy_((dk if over == "k" else dv)[l])
        b.kv.step_layer(l, new if over == "k" else dk[l], new if over == "v" else dv[l], dq[l], 1.0 / math.sqrt(D), out)
        outs.append(out)
    assert b.kv.status() == b.tide.OK
    for l in range(LAYERS):
        ref_o, ref_l = cbuild.attend_paged(b.orc.layer(l), rows, q[l], 1.0 / math.sqrt(D))
        H.check_outputs(H.from_dev(outs[l]), ref_l.astype(np.float32), ref_o, ref_l, f"layer {l}")
    b.same_bits()
    b.kv.close()


@pytest.mark.parametrize("geom", [(28, 4, 128, 16), (8, 2, 64, 32)])
@pytest.mark.parametrize("queries", [1, 40])
@pytest.mark.parametrize("which", ["fork", "write", "streams"])
def test_attention_right_behind_a_layer_sees_its_rows(geom, queries, which):
    """All queued without waiting: a step, other tasks' writers between its begin and its layers (or on the stream that the
    layers do not run on), and behind every layer attention of the step's rows, by one query (the decode kernel) or the last 40
    (tcgen05)."""
    HQ, HKV, D, S = geom
    prefix = [50 + 131 * i for i in range(40)] + [9000]
    b = Both(geom, prefix, 4)
    torch, kv, orc = b.torch, b.kv, b.orc
    n, scale = len(prefix), 1.0 / math.sqrt(D)
    sa, sb = (torch.cuda.Stream(), torch.cuda.Stream()) if which == "streams" else (None, None)
    kv.alloc(n + 3)                                           # no task of a step
    extra = [H.to_dev(x, torch) for x in (b.rows(700)[0], b.rows(700)[0])]
    kv.append([n + 3], [0, 100], *extra)
    for r in range(3 if queries == 1 else 1):
        k, v = b.rows(n), b.rows(n)
        q = np.stack([inputs.normal_bf16(b.rng, (n, HQ, D)) for _ in range(LAYERS)])
        q2 = np.stack([inputs.normal_bf16(b.rng, (n * queries, HQ, D)) for _ in range(LAYERS)])
        ip = np.arange(n + 1, dtype=np.int32)
        orc.append(b.ids, ip, k, v)
        rows = [(t, 1, orc.task_len(t)) for t in b.ids]
        rows2 = [(t, queries, orc.task_len(t)) for t in b.ids]
        dk, dv, dq, dq2 = (H.to_dev(x, torch) for x in (k, v, q, q2))
        out, out2 = torch.zeros_like(dq), torch.zeros_like(dq2)
        lse, lse2 = (torch.zeros(x.shape[:3], dtype=torch.float32, device="cuda") for x in (dq, dq2))
        torch.cuda.synchronize()

        def writer():
            if which == "fork":
                kv.fork(0, n + r)
            elif which == "write":
                kv.write(1, [n + 3], [0, 90], *extra)
            else:
                kv.write(1, [n + 3], [0, 90], *extra, stream=sa)
        kv.step_begin(rows, stream=sa)
        writer()
        if sb:
            sb.wait_stream(sa)
        for l in range(LAYERS):
            kv.step_layer(l, dk[l], dv[l], dq[l], scale, out[l], lse[l], stream=sb)
            if l == 1 and which != "fork":
                writer()
            kv.attend(rows2, dq2[l], scale, out2[l], lse2[l], layer=l, stream=sb)
        torch.cuda.synchronize()
        assert kv.status() == b.tide.OK
        for l in range(LAYERS):
            for got, gl, qq, rr, what in ((out, lse, q, rows, "layer"), (out2, lse2, q2, rows2, "attention behind layer")):
                ref_o, ref_l = cbuild.attend_paged(orc.layer(l), rr, qq[l], scale)
                H.check_outputs(H.from_dev(got[l]), gl[l].cpu().numpy(), ref_o, ref_l, f"step {r}, {what} {l}")
    b.same_bits()
    kv.close()


@pytest.mark.parametrize("geom", [(28, 4, 128, 16), (8, 2, 64, 16)])
def test_rows_are_in_the_cache_when_a_wait_has_run_out(geom):
    prefix = [5000, 3, 700, 1500, 64, 9000] + [130 + 7 * i for i in range(40)]
    b = Both(geom, prefix, 4)
    b.kv.tune(b.tide.TUNE_WAIT_LIMIT_US, 2000)

    def between(l):
        if l == 1:
            b.kv.tune(b.tide.TUNE_DROP_FIRST_STAGE, 1)        # this layer's launch: one block gives up, the next layer's starts no item

    b.step([1] * len(prefix), between, check=False)
    assert b.kv.status() == b.tide.ERR_DEVICE_TIMEOUT
    b.kv.tune(b.tide.TUNE_WAIT_LIMIT_US, 2_000_000)
    b.same_bits()
    b.step([2] * len(prefix))
    b.same_bits()
    b.kv.close()


@pytest.mark.parametrize("geom,n,prefix", [((28, 4, 128, 16), 400, 2000), ((8, 2, 64, 32), 1200, 1000)])
def test_the_block_that_gives_up_and_items_not_started_write_their_rows(geom, n, prefix):
    """Every row is one piece, longer than the ring: the block that gives up (on its first item) has not come to its row's new
    position.  The next layer finds the status word set, which keeps its items - several per resident block - from being
    started.  Bits are compared on the device."""
    import torch
    from paper_2608_10402_b200 import tide
    HQ, HKV, D, S = geom
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n)
    rows = lambda *shape: torch.randn(shape, device="cuda", generator=gen).to(torch.bfloat16)
    length = [prefix + i % 7 for i in range(n)]
    most = (prefix + 10 + S - 1) // S
    layers, pages = 2, n * most
    kv = tide.TideKV(HQ, HKV, D, S, pages, n, most, n, 4096, free_order=np.random.default_rng(n).permutation(pages).astype(np.int32), num_layers=layers)
    old = [(rows(prefix + 6, HKV, D), rows(prefix + 6, HKV, D)) for _ in range(layers)]     # every task begins with the same tokens
    for t in range(n):
        kv.alloc(t)
        kv.extend([t], [0, length[t]])
        for l in range(layers):
            kv.write(l, [t], [0, length[t]], old[l][0][:length[t]], old[l][1][:length[t]])
    new_k, new_v, q = rows(layers, n, HKV, D), rows(layers, n, HKV, D), rows(layers, n, HQ, D)
    out = torch.zeros_like(q)
    assert kv.status() == tide.OK
    kv.tune(tide.TUNE_WAIT_LIMIT_US, 2000)
    kv.step_begin([(t, 1, length[t] + 1) for t in range(n)])
    kv.tune(tide.TUNE_DROP_FIRST_STAGE, 1)
    for l in range(layers):
        kv.step_layer(l, new_k[l], new_v[l], q[l], 1.0 / math.sqrt(D), out[l])
    assert kv.last_plan()["decode_items"] == n * HKV           # one piece a row
    assert kv.status() == tide.ERR_DEVICE_TIMEOUT
    left_out = [int((o.view(n, HKV, -1) == 0).all(-1).sum()) for o in out]     # items that were not started
    assert left_out[0] == 0                                    # the 2 ms are longer than the others take
    # the second layer's blocks that start beside the first, two on an SM, may have begun one item each before the word was set
    assert n * HKV - left_out[1] <= 2 * torch.cuda.get_device_properties(0).multi_processor_count, left_out
    for l in range(layers):
        for t in range(n):
            k, v = kv.read(t, layer=l)
            for got, before, row in ((k, old[l][0], new_k[l, t]), (v, old[l][1], new_v[l, t])):
                got = got.view(torch.bfloat16)
                assert torch.equal(got[-1], row) and torch.equal(got[:-1], before[:length[t]]), (l, t)
    kv.close()
