"""The GEMM kernel's tall tiles (two row tiles high), forced through the shape knob: one row tile only, an odd number of
them, ragged edges in every dimension, with the shrink inside the kernel and with the launch ahead of it."""
import numpy as np
import pytest

import oracle
from paper_2608_15241_b200 import workloads as wl

from gpu_util import Site

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fuse", ["1", "0"])
@pytest.mark.parametrize("kw", [dict(T=128, d_in=264, d_out=264), dict(T=257, d_in=1032, d_out=520),
                                dict(T=333, d_in=320, d_out=456, shuffled=True), dict(T=384, d_in=64, d_out=2056),
                                dict(T=700, d_in=520, d_out=8192), dict(T=1300, d_in=1032, d_out=4104, shuffled=True)])
def test_tall_tiles_against_oracle(kw, fuse, monkeypatch):
    monkeypatch.setenv("LML_GEMM_SPLIT", "512x1")
    monkeypatch.setenv("LML_FUSE_SHRINK", fuse)
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


@pytest.mark.parametrize("T", [130, 300, 700])
def test_tall_tiles_of_several_projections(T, monkeypatch):
    """Tiles numbered through three projections of unequal width, an odd number of row tiles among them."""
    import torch
    from paper_2608_15241_b200 import binding as b
    from paper_2608_15241_b200.binding import Table
    from gpu_util import to_bits, to_dev
    monkeypatch.setenv("LML_GEMM_SPLIT", "512x1")
    K, Ns, ranks = 520, (264, 1000, 136), (4, 33, 64)
    x = wl.normal_bf16(9, 1, (T, K), 1.0)
    tok = np.random.default_rng(T).integers(-1, len(ranks), size=T).astype(np.int32)
    tables, W, ents = [], [], []
    for p, N in enumerate(Ns):
        W.append(wl.normal_bf16(9, 10 + p, (N, K), 0.02))
        ents.append(wl.make_entries(9 + p, K, N, [(a, 1, r, 2.0) for a, r in enumerate(ranks)]))
        tables.append(Table(K, N, len(ranks)))
        for e in ents[p]:
            tables[p].register_adapter(e.adapter_id, 1, to_dev(e.A), to_dev(e.B), e.scale)
    ys = b.multi_projection(tables, to_dev(x), [to_dev(w) for w in W], torch.from_numpy(tok).cuda())
    torch.cuda.synchronize()
    for p in range(len(Ns)):
        ref, _ = oracle.forward(x, W[p], ents[p], np.arange(T + 1, dtype=np.int32), tok)
        r = oracle.compare(to_bits(ys[p]), ref)
        assert r["ok"] and tables[p].device_status() == 0, (p, r)
        tables[p].close()
