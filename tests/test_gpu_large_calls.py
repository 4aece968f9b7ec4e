"""Calls beyond the sizes of the other tests, on narrow layers and sampled rows: many slots in every row tile (several passes
of bind_shrink through one ring), more row tiles than a slab holds, more segments than the kernels look up in shared memory."""
import numpy as np
import pytest

import oracle
from paper_2608_15241_b200 import workloads as wl

from gpu_util import Guarded, to_bits, to_dev

pytestmark = pytest.mark.gpu


def _site(K, N, ranks, seed=17, std=0.05):
    from paper_2608_15241_b200.binding import Table
    entries = wl.make_entries(seed, K, N, [(a, 1, r, 2.0) for a, r in enumerate(ranks)], std=std)
    tbl = Table(K, N, len(ranks))
    for e in entries:
        tbl.register_adapter(e.adapter_id, 1, to_dev(e.A), to_dev(e.B), e.scale)
    return tbl, entries, wl.normal_bf16(seed, 2, (N, K), std)


def _sample(T, seed=0):
    """a row of every 128, those around the slabs' border and the last"""
    rng = np.random.default_rng(seed)
    pos = {int(min(T - 1, t0 + rng.integers(0, 128))) for t0 in range(0, T, 128)}
    pos.update(p for p in (0, 65535, 65536, T - 1) if 0 <= p < T)
    return np.array(sorted(pos), np.int32)


def _check(y, x, W, entries, entry, pos):
    ref, _ = oracle.forward(x[pos], W, entries, np.arange(len(pos) + 1, dtype=np.int32), entry[pos])
    r = oracle.compare(to_bits(y)[pos], ref)
    assert r["ok"], r


@pytest.mark.parametrize("T", [300, 5000])
@pytest.mark.parametrize("ranks", [(16,), (16, 9), (33,), (64, 4), (16,) * 18])
def test_few_chunks_on_many_laps_of_the_ring(T, ranks):
    """Passes of one, two, three and five chunks, and of two after full ones, over 129 k-blocks: fewer chunks than bind_shrink has warps that
    copy them, and a ring that goes round many times.  (Adapters of N(0, 0.02): u is 2 x.A, of size 2 sqrt(8200) 0.02 = 3.6, and its rounding to
    bf16, 2^-9 of it in the mean, reaches y through at most 64 entries of B: 3.6 2^-9 0.02 8 = 1.1e-3, a ninth of the tolerance.)"""
    import torch
    K, N = 8200, 136
    tbl, entries, W = _site(K, N, ranks, std=0.02)
    x = wl.normal_bf16(31, 1, (T, K), 1.0)
    entry = np.random.default_rng(T).integers(-1, len(ranks), size=T).astype(np.int32)
    tok = torch.from_numpy(entry).cuda()
    ys = [tbl.lora_mixed_linear_tokens(to_dev(x), to_dev(W), tok) for _ in range(3)]
    torch.cuda.synchronize()
    assert tbl.device_status() == 0
    _check(ys[0], x, W, entries, entry, _sample(T))
    assert all(torch.equal(ys[0], y) for y in ys[1:])
    tbl.close()


@pytest.mark.parametrize("T", [5000, 9600])
@pytest.mark.parametrize("ranks", [(64, 33, 16, 8) * 5, (64,) * 17 + (1,), (4,) * 40])
def test_many_slots_in_every_row_tile(T, ranks):
    import torch
    K, N = 264, 136
    tbl, entries, W = _site(K, N, ranks)
    x = wl.normal_bf16(1, 1, (T, K), 1.0)
    entry = np.random.default_rng(T).integers(-1, len(ranks), size=T).astype(np.int32)
    ids, xd, Wd = torch.from_numpy(entry).cuda(), to_dev(x), to_dev(W)
    y = tbl.lora_mixed_linear_tokens(xd, Wd, ids)
    again = tbl.lora_mixed_linear_tokens(xd, Wd, ids)
    torch.cuda.synchronize()
    assert tbl.device_status() == 0 and torch.equal(y.view(torch.int16), again.view(torch.int16))
    _check(y, x, W, entries, entry, _sample(T))
    perm, so, se = tbl.segment_tokens(ids)
    _check(tbl.lora_mixed_linear(xd, Wd, so, se, perm=perm), x, W, entries, entry, _sample(T, 1))
    assert tbl.device_status() == 0
    tbl.close()


def test_more_row_tiles_than_a_slab():
    import torch
    from paper_2608_15241_b200 import binding as b
    T, K, N, ranks = 66_000, 72, 40, (4, 16, 33)
    tbl, entries, W = _site(K, N, ranks)
    x = wl.normal_bf16(1, 1, (T, K), 1.0)
    entry = np.random.default_rng(3).integers(-1, len(ranks), size=T).astype(np.int32)
    pos = _sample(T)
    ids, xd, Wd = torch.from_numpy(entry).cuda(), to_dev(x), to_dev(W)
    gy, gws = Guarded(T * N * 2), Guarded(b.lml_tokens_workspace_bytes(tbl.handle, T))
    y = gy.view(torch.bfloat16, (T, N))
    tbl.lora_mixed_linear_tokens(xd, Wd, ids, y=y, workspace=gws.payload)
    torch.cuda.synchronize()
    assert gy.intact() and gws.intact()
    _check(y, x, W, entries, entry, pos)
    perm, so, se = tbl.segment_tokens(ids)
    _check(tbl.lora_mixed_linear(xd, Wd, so, se, perm=perm), x, W, entries, entry, pos)
    # segments in order (one of them across the border), one binding and two
    cuts = np.array([0, 20_000, 65_500, 65_600, T], np.int32)
    ea, eb = np.array([0, -1, 2, 1], np.int32), np.array([1, 2, 2, -1], np.int32)
    so, sa, sb = (torch.from_numpy(a).cuda() for a in (cuts, ea, eb))
    by_row = lambda e: np.repeat(e, np.diff(cuts)).astype(np.int32)  # noqa: E731
    _check(tbl.lora_mixed_linear(xd, Wd, so, sa), x, W, entries, by_row(ea), pos)
    ya, yb = tbl.lora_mixed_linear_dual(xd, Wd, so, sa, sb)
    _check(ya, x, W, entries, by_row(ea), pos)
    _check(yb, x, W, entries, by_row(eb), pos)
    assert tbl.device_status() == 0
    tbl.close()


@pytest.mark.parametrize("T", [40, 700, 2000])
@pytest.mark.parametrize("shuffled", [False, True])
def test_more_segments_than_the_kernels_keep_in_shared_memory(T, shuffled):
    import torch
    from paper_2608_15241_b200 import binding as b
    K, N, G, ranks = 264, 136, 300, (4, 16, 33, 64)
    tbl, entries, W = _site(K, N, ranks)
    rng = np.random.default_rng(T)
    x = wl.normal_bf16(1, 1, (T, K), 1.0)
    so = np.concatenate([[0], np.sort(rng.integers(0, T + 1, size=G - 1)), [T]]).astype(np.int32)   # empty segments among them
    se = rng.integers(-1, len(ranks), size=G).astype(np.int32)
    perm = rng.permutation(T).astype(np.int32) if shuffled else None
    entry = np.empty(T, np.int32)
    entry[perm if shuffled else np.arange(T)] = np.repeat(se, np.diff(so))
    dev = lambda a: None if a is None else torch.from_numpy(a).cuda()  # noqa: E731
    y = tbl.lora_mixed_linear(to_dev(x), to_dev(W), dev(so), dev(se), perm=dev(perm))
    torch.cuda.synchronize()
    _check(y, x, W, entries, entry, np.arange(T, dtype=np.int32))
    assert tbl.device_status() == 0
    bad = so.copy()
    bad[150] = T + 5                     # not monotone: every row gets base output
    y = tbl.lora_mixed_linear(to_dev(x), to_dev(W), dev(bad), dev(se), perm=dev(perm))
    torch.cuda.synchronize()
    _check(y, x, W, entries, np.full(T, -1, np.int32), np.arange(T, dtype=np.int32))
    assert tbl.device_status() & b.FLAG_BAD_OFFSETS
    tbl.close()
