"""An adapter whose B holds Inf or NaN concerns its own tokens only: y[t] is defined by the entry of token t alone.  Beside it,
tokens of other adapters and of none keep their bits; its own rows get Inf or NaN in the columns whose row of B is not finite, by
the sign of u, and keep their bits elsewhere.  Every form of the GEMM path, with the decode kernel as a cross-check."""
import numpy as np
import pytest

from paper_2608_15241_b200 import workloads as wl

from gpu_util import to_bits, to_dev

pytestmark = pytest.mark.gpu

RANKS = (4, 33, 16, 64)
BROKEN = 1
INF, NINF, NAN = 0x7f80, 0xff80, 0x7fc0


def _adapters(K, N, seed):
    out = []
    for a, r in enumerate(RANKS):
        A, B = wl.normal_bf16(seed, 10 + a, (r, K), 0.05), wl.normal_bf16(seed, 30 + a, (N, r), 0.05)
        out.append((A, B))
    return out


def _break(B, r):
    """(B with entries that are not finite, the same with zeros there, {row of B: (column, value)})"""
    N = B.shape[0]
    where = {5: (0, INF), 9: (r - 1, NINF), 17: (r // 2, NAN), N - 1: (1, INF)}
    broken, clean = B.copy(), B.copy()
    for n, (j, v) in where.items():
        broken[n, j], clean[n, j] = v, 0
    return broken, clean, where


def _call(form, tables, x, Ws, entry):
    """outputs [(y, entry per row, projection)] of one call of the form"""
    import torch
    from paper_2608_15241_b200 import binding as b
    ids = torch.from_numpy(entry).cuda()
    T = len(entry)
    if form == "tokens":
        return [(tables[0].lora_mixed_linear_tokens(x, Ws[0], ids), entry, 0)]
    if form == "multi":
        return [(y, entry, p) for p, y in enumerate(b.multi_projection(tables, x, Ws, ids))]
    cuts = np.flatnonzero(np.diff(entry)) + 1
    so = torch.from_numpy(np.concatenate([[0], cuts, [T]]).astype(np.int32)).cuda()
    se = entry[np.concatenate([[0], cuts])].astype(np.int32)
    if form == "segments":
        return [(tables[0].lora_mixed_linear(x, Ws[0], so, torch.from_numpy(se).cuda()), entry, 0)]
    if form == "perm":
        perm, po, pe = wl.group_tokens(entry, len(RANKS))
        y = tables[0].lora_mixed_linear(x, Ws[0], torch.from_numpy(po).cuda(), torch.from_numpy(pe).cuda(), perm=torch.from_numpy(perm).cuda())
        return [(y, entry, 0)]
    se_b = np.where(np.arange(len(se)) % 3 == 0, se, np.roll(se, 1)).astype(np.int32)
    ya, yb = tables[0].lora_mixed_linear_dual(x, Ws[0], so, torch.from_numpy(se).cuda(), torch.from_numpy(se_b).cuda())
    return [(ya, entry, 0), (yb, np.repeat(se_b, np.diff(np.concatenate([[0], cuts, [T]]))).astype(np.int32), 0)]


@pytest.mark.parametrize("form,T,K,Ns", [
    ("tokens", 12, 264, (136,)), ("tokens", 70, 1032, (264,)), ("tokens", 129, 2048, (520,)), ("tokens", 700, 520, (8200,)),
    ("tokens", 2500, 264, (2056,)), ("multi", 40, 520, (264, 136)), ("multi", 48, 2048, (2056, 1032)), ("multi", 300, 520, (264, 1000)),
    ("segments", 200, 1032, (520,)), ("segments", 700, 520, (8192,)), ("segments", 2100, 264, (5000,)), ("perm", 700, 520, (8192,)),
    ("dual", 96, 2048, (520,)), ("dual", 600, 264, (8200,)), ("dual", 2100, 512, (5000,))])
def test_rows_of_other_slots_keep_their_bits(form, T, K, Ns):
    import torch
    from paper_2608_15241_b200.binding import Table
    rng = np.random.default_rng(T)
    runs = form in ("segments", "dual")
    entry = rng.integers(-1, len(RANKS), size=12 if runs else T).astype(np.int32)
    entry[3] = BROKEN
    if runs:
        cuts = np.sort(rng.choice(np.arange(1, T), size=11, replace=False))
        entry = np.repeat(entry, np.diff(np.concatenate([[0], cuts, [T]]))).astype(np.int32)
    x_bits = wl.normal_bf16(7, 1, (T, K), 1.0)
    x = to_dev(x_bits)
    Ws = [to_dev(wl.normal_bf16(7, 2 + p, (N, K), 0.05)) for p, N in enumerate(Ns)]
    ads = [_adapters(K, N, 50 + p) for p, N in enumerate(Ns)]
    got = {}
    for kind in ("clean", "broken", "clean again"):
        if kind != "clean again":
            tables = [Table(K, N, len(RANKS)) for N in Ns]
        else:       # the broken version is retired and a sound one takes its slot
            for t in tables:
                t.retire_version(BROKEN, 1)
        for t, ad in zip(tables, ads):
            for a, (A, B) in enumerate(ad):
                if kind == "clean again" and a != BROKEN:
                    continue
                if a == BROKEN:
                    broken, clean, _ = _break(B, RANKS[a])
                    B = broken if kind == "broken" else clean
                assert t.register_adapter(a, 2 if kind == "clean again" else 1, to_dev(A), to_dev(B), 1.5) == a
        got[kind] = _call(form, tables, x, Ws, entry)
        torch.cuda.synchronize()
        assert all(t.device_status() == 0 for t in tables)
        if kind != "broken":
            for t in tables if kind == "clean again" else []:
                t.close()
    xf = wl.bf16_bits_to_f64(x_bits)
    for (yc, _, _), (yb, ent, p), (y2, _, _) in zip(got["clean"], got["broken"], got["clean again"]):
        yc, yb, y2 = to_bits(yc), to_bits(yb), to_bits(y2)
        assert np.isfinite(wl.bf16_bits_to_f64(yc)).all()
        assert np.array_equal(yc, y2)
        own = ent == BROKEN
        assert own.any() and np.array_equal(yb[~own], yc[~own])
        where = _break(ads[p][BROKEN][1], RANKS[BROKEN])[2]
        rest = np.setdiff1d(np.arange(Ns[p]), list(where))
        assert np.array_equal(yb[own][:, rest], yc[own][:, rest])
        u = xf[own] @ wl.bf16_bits_to_f64(ads[p][BROKEN][0]).T
        for n, (j, v) in where.items():
            col = wl.bf16_bits_to_f64(yb[own][:, n])
            sure = np.abs(u[:, j]) > 1e-2       # the sign of u is beyond its rounding
            if v == NAN:
                assert np.isnan(col).all()
            else:
                assert np.array_equal(np.sign(col[sure]), np.sign(u[sure, j]) * (1 if v == INF else -1)) and np.isinf(col[sure]).all()
