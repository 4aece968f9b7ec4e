"""The GEMM of CTA pairs at every width of its tiles, forced through the shape knob: one row tile (the second CTA's rows lie outside x),
an odd number of row tiles, two tiles to a pair and many, panels of rows, chunks that only one of a pair's row tiles uses; against the
oracle."""
import numpy as np
import pytest

import oracle
from paper_2608_15241_b200 import workloads as wl

from gpu_util import Site

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width", [64, 96, 128, 160, 192, 224, 256])
@pytest.mark.parametrize("kw", [dict(T=128, d_in=72, d_out=520), dict(T=129, d_in=584, d_out=264), dict(T=700, d_in=320, d_out=3000, shuffled=True)])
def test_every_width_against_oracle(width, kw, monkeypatch):
    monkeypatch.setenv("LML_GEMM_SPLIT", f"{width}p")
    w = wl.ragged(ranks=(4, 16, 1, 33, 64), **kw)
    site = Site(w)
    y, flags = site.run()
    y2, _ = site.run()
    yb, fb = site.run(seg_offsets=[0, w.T], raw_slot_ids=[-1])
    site.close()
    ref, _ = oracle.forward_workload(w)
    r = oracle.compare(y, ref)
    assert flags == 0 and r["ok"], r
    assert np.array_equal(y, y2)
    refb, _ = oracle.forward(w.x, w.W0, w.entries, np.array([0, w.T], np.int32), np.array([-1], np.int32), w.perm)
    assert fb == 0 and oracle.compare(yb, refb)["ok"]


@pytest.mark.parametrize("width,T,d_in,d_out", [(96, 2300, 64, 3240), (160, 2300, 64, 5160), (160, 2300, 136, 5160), (224, 2300, 128, 7192),
                                                (256, 60000, 64, 280), (256, 60000, 256, 280)])
@pytest.mark.parametrize("shuffled", [False, True])
def test_many_tiles_to_a_pair(width, T, d_in, d_out, shuffled, monkeypatch):
    """Four tiles and more to each of the 74 pairs, an odd number of 32-column chunks stored in each (at 256 columns in the second half of
    the tiles, of which y holds one chunk), and so little K that the epilogue is what the tiles wait for: the staging buffers, the two
    accumulators and the two lists of chunks are used again and again."""
    monkeypatch.setenv("LML_GEMM_SPLIT", f"{width}p")
    w = wl.ragged(T=T, d_in=d_in, d_out=d_out, ranks=(4, 16, 1, 33, 64), shuffled=shuffled)
    assert (w.T + 255) // 256 * ((d_out + width - 1) // width) >= 4 * 74
    site = Site(w)
    y, flags = site.run()
    again = [site.run()[0] for _ in range(3)]
    yb, fb = site.run(seg_offsets=[0, w.T], raw_slot_ids=[-1])
    site.close()
    ref, _ = oracle.forward_workload(w)
    r = oracle.compare(y, ref)
    assert flags == 0 and r["ok"], r
    assert all(np.array_equal(y, a) for a in again)
    refb, _ = oracle.forward(w.x, w.W0, w.entries, np.array([0, w.T], np.int32), np.array([-1], np.int32), w.perm)
    assert fb == 0 and oracle.compare(yb, refb)["ok"]


def test_several_panels_of_rows(monkeypatch):
    """More x than a panel holds (48 MB): 3500 rows of 8200 columns in two panels, the second shorter; sampled rows."""
    monkeypatch.setenv("LML_GEMM_SPLIT", "256p")
    w = wl.ragged(T=3500, d_in=8200, d_out=264, ranks=(16, 8))
    site = Site(w)
    y, flags = site.run()
    site.close()
    from gpu_util import sample_positions_every_tile
    pos = sample_positions_every_tile(w, 60)
    ref, _ = oracle.forward(w.x, w.W0, w.entries, w.seg_offsets, w.seg_entry, w.perm, positions=pos)
    rows = pos if w.perm is None else w.perm[pos]
    r = oracle.compare(y[rows], ref[rows])
    assert flags == 0 and r["ok"], r


@pytest.mark.parametrize("T", [17, 48])
def test_u_of_three_values_does_not_take_pairs(T, monkeypatch):
    """A call of several projections at 17 - 48 tokens multiplies u as three bf16 values, which the pair kernel has no place for: with pairs
    asked for it runs on whole-K tiles, and keeps its bits."""
    import torch
    from paper_2608_15241_b200 import binding as b
    from paper_2608_15241_b200.binding import Table
    from gpu_util import to_bits, to_dev
    K, Ns, ranks = 520, (264, 1000), (4, 33, 64)
    x, tok = wl.normal_bf16(9, 1, (T, K), 1.0), np.random.default_rng(T).integers(-1, len(ranks), size=T).astype(np.int32)
    W = [wl.normal_bf16(9, 10 + p, (N, K), 0.02) for p, N in enumerate(Ns)]
    ents = [wl.make_entries(9 + p, K, N, [(a, 1, r, 2.0) for a, r in enumerate(ranks)]) for p, N in enumerate(Ns)]
    out = []
    for shape in ("0", "128p"):
        monkeypatch.setenv("LML_GEMM_SPLIT", shape)
        tables = [Table(K, N, len(ranks)) for N in Ns]
        for t, es in zip(tables, ents):
            for e in es:
                t.register_adapter(e.adapter_id, 1, to_dev(e.A), to_dev(e.B), e.scale)
        ys = b.multi_projection(tables, to_dev(x), [to_dev(w) for w in W], torch.from_numpy(tok).cuda())
        torch.cuda.synchronize()
        assert all(t.device_status() == 0 for t in tables)
        out.append([to_bits(y) for y in ys])
        for t in tables:
            t.close()
    for p in range(len(Ns)):
        assert np.array_equal(out[0][p], out[1][p]), p
        ref, _ = oracle.forward(x, W[p], ents[p], np.arange(T + 1, dtype=np.int32), tok)
        assert oracle.compare(out[1][p], ref)["ok"], p


def test_whole_k_tiles_of_every_form_agree_bit_for_bit(monkeypatch):
    """Which whole-K tiles a call takes follows from estimates; its bits do not: single tiles, tall tiles and pairs of every width add up in
    one order.  So does a dual call's first output, although a dual call takes no pairs."""
    import torch
    from gpu_util import to_bits
    w = wl.ragged(T=700, d_in=1032, d_out=1000, ranks=(4, 16, 1, 33, 64))
    monkeypatch.setenv("LML_FUSE_SHRINK", "0")   # (inside the GEMM kernel u is summed in another order)
    ys = {}
    for shape in ("64x1", "128x1", "256x1", "512x1", "64p", "160p", "256p", None):
        if shape:
            monkeypatch.setenv("LML_GEMM_SPLIT", shape)
        else:
            monkeypatch.delenv("LML_GEMM_SPLIT")
        site = Site(w)
        ys[shape], flags = site.run()
        assert flags == 0
        if shape in ("256x1", None):
            so, ids = torch.from_numpy(w.seg_offsets).cuda(), torch.from_numpy(site.slot_ids()).cuda()
            ys["dual", shape] = to_bits(site.table.lora_mixed_linear_dual(site.x, site.W0, so, ids, ids.flip(0).contiguous())[0])
        site.close()
    ref, _ = oracle.forward_workload(w)
    assert oracle.compare(ys["64x1"], ref)["ok"]
    for shape, y in ys.items():
        assert np.array_equal(y, ys["64x1"]), shape
