"""Calls back to back on one stream, one workspace and one table, nothing waited for in between: every call sees the x, the ids
and the plan of its own binding, and a captured call replayed sees what stream work has written since the last replay.  Sizes
are those whose GEMM starts while the work before the call is still running, and larger ones whose GEMM does not."""
import numpy as np
import pytest

from paper_2608_15241_b200 import workloads as wl

from gpu_util import to_bits, to_dev

pytestmark = pytest.mark.gpu

SIZES = [(40, 2048, 520), (128, 1032, 264), (200, 2048, 1000), (2500, 520, 264)]


def _site(K, N, seed=3, ranks=(4, 16, 33, 8)):
    from paper_2608_15241_b200.binding import Table
    tbl = Table(K, N, len(ranks))
    for a, r in enumerate(ranks):
        tbl.register_adapter(a, 1, to_dev(wl.normal_bf16(seed, 10 + a, (r, K), 0.05)), to_dev(wl.normal_bf16(seed, 30 + a, (N, r), 0.05)), 1.5)
    return tbl, to_dev(wl.normal_bf16(seed, 2, (N, K), 0.05))


def _ids(T, seed, n=4):
    import torch
    rng = np.random.default_rng(seed)
    some = rng.permutation(n)[:1 + seed % n]             # few slots one time, all of them another: the plans differ in length
    ids = rng.choice(np.concatenate([some, [-1]]), size=T).astype(np.int32)
    return torch.from_numpy(ids).cuda()


@pytest.mark.parametrize("T,K,N", SIZES)
def test_calls_in_a_row_each_see_their_own_binding(T, K, N):
    import torch
    from paper_2608_15241_b200 import binding as b
    tbl, W = _site(K, N)
    xs = [to_dev(wl.normal_bf16(s, 1, (T, K), 1.0)) for s in range(6)]
    ids = [_ids(T, s) for s in range(6)]
    ws = torch.empty(max(256, b.lml_tokens_workspace_bytes(tbl.handle, T)), dtype=torch.uint8, device="cuda")
    want = []
    for x, i in zip(xs, ids):
        want.append(to_bits(tbl.lora_mixed_linear_tokens(x, W, i, workspace=ws)))
        torch.cuda.synchronize()
    for _ in range(5):
        got = [tbl.lora_mixed_linear_tokens(x, W, i, workspace=ws) for x, i in zip(xs, ids)]
        torch.cuda.synchronize()
        assert all(np.array_equal(to_bits(g), w) for g, w in zip(got, want))
    assert tbl.device_status() == 0
    tbl.close()


@pytest.mark.parametrize("T,K,N", SIZES)
def test_a_replayed_call_reads_what_was_written_since(T, K, N):
    import torch
    from paper_2608_15241_b200 import binding as b
    tbl, W = _site(K, N)
    x, i = torch.empty(T, K, dtype=torch.bfloat16, device="cuda"), torch.empty(T, dtype=torch.int32, device="cuda")
    y = torch.empty(T, N, dtype=torch.bfloat16, device="cuda")
    ws = torch.empty(max(256, b.lml_tokens_workspace_bytes(tbl.handle, T)), dtype=torch.uint8, device="cuda")
    xs = [to_dev(wl.normal_bf16(s, 1, (T, K), 1.0)) for s in range(5)]
    ids = [_ids(T, s) for s in range(5)]
    want = []
    for a, c in zip(xs, ids):
        want.append(to_bits(tbl.lora_mixed_linear_tokens(a, W, c, workspace=ws)))
    x.copy_(xs[0]); i.copy_(ids[0])
    tbl.lora_mixed_linear_tokens(x, W, i, y=y, workspace=ws)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        tbl.lora_mixed_linear_tokens(x, W, i, y=y, workspace=ws)
    out = []
    for _ in range(3):
        for a, c in zip(xs, ids):                        # the writes and the replay in stream order, the host waits for neither
            x.copy_(a); i.copy_(c)
            graph.replay()
            out.append(y.clone())
    torch.cuda.synchronize()
    assert all(np.array_equal(to_bits(o), want[k % 5]) for k, o in enumerate(out))
    assert tbl.device_status() == 0
    del graph
    tbl.close()


@pytest.mark.parametrize("T", [40, 128, 200, 1500])
def test_a_call_reads_the_x_that_the_call_before_it_wrote(T):
    import torch
    K = 2048
    tbl, W = _site(K, K)
    ids = [_ids(T, s) for s in range(4)]

    def chain(wait):
        x = to_dev(wl.normal_bf16(1, 1, (T, K), 1.0))
        for s in range(8):
            x = tbl.lora_mixed_linear_tokens(x, W, ids[s % 4])
            if wait:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        return to_bits(x)

    want = chain(True)
    assert all(np.array_equal(chain(False), want) for _ in range(4))
    assert tbl.device_status() == 0
    tbl.close()


def test_a_call_behind_work_that_releases_its_dependents_early_and_runs_on():
    """The segmentation kernel lets the kernels behind it start at once and then works on millions of tokens for longer than the
    GEMM polls for x: the call behind it waits as long as that takes, with all its limits counted from there."""
    import torch
    T, K, N = 40, 2048, 520
    tbl, W = _site(K, N)
    x, ids = to_dev(wl.normal_bf16(1, 1, (T, K), 1.0)), _ids(T, 3)
    want = to_bits(tbl.lora_mixed_linear_tokens(x, W, ids))
    many = _ids(4_000_000, 3)
    torch.cuda.synchronize()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record()
    tbl.segment_tokens(many)
    b.record()
    torch.cuda.synchronize()
    print("segmentation", a.elapsed_time(b), "ms")
    for _ in range(3):
        tbl.segment_tokens(many)
        y = tbl.lora_mixed_linear_tokens(x, W, ids)
        torch.cuda.synchronize()
        assert np.array_equal(to_bits(y), want)
    assert tbl.device_status() == 0
    tbl.close()
