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
