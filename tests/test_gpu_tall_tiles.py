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
