"""The work a multi-agent runtime has this layer do, as cases whose time and results can be compared.

Most cases are one pass over the seven projections of a decoder layer (q, k, v, o, gate, up, down), the
unit in which a model calls the layer: q/k/v and gate/up read the same activations, the seven weights
together are larger than L2, so every weight comes out of HBM as it does in a model of many layers.
Sizes are those of this repository's workloads (4096 / 11008, ranks 8 ... 64, 5 or 18 resident entries,
Zipf(1.1) binding) and generic ones beside them (other widths, narrower k and v).

A case:
  kind      layer    token-form calls: one slot id per token, the two multi-projection groups in one call each
            segments the batch arrives as contiguous segments (what a prefill scheduler hands over)
            publish  a new version of one adapter is registered and published at every projection, then the
                     layer runs by adapter id, so its tokens see the version that has just been published
            dual     the layer under two bindings at once (the old and the staged version of an adapter)
            train    one training pass: forward, dx and the adapter gradients of every projection
            small    one projection of a small model, called on its own
            host     one projection called on host buffers, the result read on the host
  tokens, hidden, ffn, kv   sizes: q, o are hidden x hidden, k and v hidden -> kv, gate and up hidden -> ffn,
            down ffn -> hidden (small and host: hidden -> ffn only)
  adapters  adapters resident; versions: how many of them are resident in a second version too
  ranks     their ranks in turn; none: the share of tokens without an adapter
  runs      0: every token draws its entry (tokens of many agents interleaved); n: the batch is n requests,
            each a run of tokens on one entry
  graph     the pass is captured once and replayed, as the decode loop of a serving runtime does
"""
from __future__ import annotations

import math
from typing import List

import numpy as np
import torch

from paper_2608_15241_b200.binding import Table, lml_multi_workspace_bytes, multi_projection

SCALE = 2.0
STD = 0.02          # of W0, A and B; x and dy are N(0, 1)
SPARE_SLOTS = 2     # room for staged versions
ZIPF = 1.1


def _case(name, kind, tokens, hidden, ffn, kv, adapters, versions, ranks, none=0.0, runs=0, graph=False):
    return dict(name=name, kind=kind, tokens=tokens, hidden=hidden, ffn=ffn, kv=kv, adapters=adapters, versions=versions,
                ranks=ranks, none=none, runs=runs, graph=graph)


def listed() -> List[dict]:
    return [
        # one agent generating alone: latency of a decode step
        _case("decode_1", "layer", 1, 4096, 11008, 4096, 16, 2, "16", graph=True),
        # four agents, two tokens each, one adapter in two versions: the usual decode step
        _case("decode_8", "layer", 8, 4096, 11008, 4096, 4, 1, "16", graph=True),
        # a crowded decode step of a model with narrow k and v; adapters of every rank, some tokens on the bare base
        _case("decode_40_mixed", "layer", 40, 5120, 13824, 1024, 8, 0, "8,16,32,64", none=0.1, graph=True),
        # a small model's projection called eagerly: launches and host work
        _case("small_64", "small", 64, 256, 256, 256, 3, 0, "4,8,8", runs=3),
        # activations in host memory, a decode step's worth
        _case("host_8", "host", 8, 4096, 4096, 4096, 4, 1, "16", runs=4),
        # the first prefill that hits a version published just before it
        _case("publish_300", "publish", 300, 4096, 11008, 4096, 4, 0, "16", runs=4),
        # a prefill chunk of many agents' tokens
        _case("chunk_128", "layer", 128, 4096, 11008, 4096, 16, 2, "16"),
        # a mixed batch of prefill chunks and decode tokens, in arrival order
        _case("batch_500_mixed", "layer", 500, 3072, 8192, 1024, 8, 0, "8,16,32,64", none=0.1),
        # post-publish prefill: a few long segments
        _case("prefill_2048", "segments", 2048, 4096, 11008, 4096, 4, 1, "16", runs=4),
        # the largest prefill batch, requests of all adapters and of none
        _case("prefill_8192_mixed", "layer", 8192, 4096, 11008, 4096, 8, 0, "8,16,32,64", none=0.1, runs=24),
        # a hot prefix recomputed under the staged version while the old one serves
        _case("dual_96", "dual", 96, 4096, 11008, 4096, 4, 1, "16", runs=4),
        # a background training batch of two adapters
        _case("train_1000", "train", 1000, 4096, 11008, 4096, 2, 0, "16", runs=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng) -> dict:
    kind = rng.choice(["layer"] * 6 + ["segments", "segments", "publish", "dual", "train", "small", "host"])
    hidden = rng.choice([2048, 2560, 3072, 4096, 4096, 4096, 5120, 8 * rng.randint(256, 640)])
    ffn = {2048: 5632, 2560: 6912, 3072: 8192, 4096: 11008, 5120: 13824}.get(hidden) or 8 * rng.randint(hidden // 4, hidden // 3)
    kv = hidden if rng.random() < 0.6 else 8 * (hidden // 32)
    most = {"layer": 8192, "segments": 8192, "publish": 2048, "dual": 2048, "train": 2048, "small": 512, "host": 2048}[kind]
    if hidden > 4096:
        most //= 2
    tokens = _log_int(rng, {"publish": 260, "train": 16, "small": 16}.get(kind, 1), most)
    if kind == "small":
        hidden, ffn = 8 * _log_int(rng, 16, 128), 8 * _log_int(rng, 16, 128)
        kv = hidden
    adapters = rng.randint(2, 16)
    case = _case("", kind, tokens, hidden, ffn, kv, adapters, rng.randint(0, 2), rng.choice(["16", "16", "8", "32", "8,16,32,64", "4,8,8"]),
                 none=rng.choice([0.0, 0.0, 0.1]), runs=rng.choice([0, 4, adapters, 24]),
                 graph=kind == "layer" and tokens <= 64 and rng.random() < 0.7)
    if kind not in ("layer",) and case["runs"] == 0:
        case["runs"] = 4
    if kind in ("publish", "train"):
        case["versions"] = 0
    if kind == "train":                                                # the adapters being trained, not all resident ones
        case["adapters"] = rng.randint(1, 4)
    del case["name"]
    return case


# ---- sizes --------------------------------------------------------------------------------------------

def _sites(case):
    """(name, d_in, d_out, which activations it reads) of every projection of the pass."""
    h, f, kv = case["hidden"], case["ffn"], case["kv"]
    if case["kind"] in ("small", "host"):
        return [("proj", h, f, 0)]
    return [("q", h, h, 0), ("k", h, kv, 0), ("v", h, kv, 0), ("o", h, h, 1),
            ("gate", h, f, 2), ("up", h, f, 2), ("down", f, h, 3)]


def _entries(case):
    """(adapter, version, rank) of every resident entry, in slot order."""
    ranks = [int(r) for r in case["ranks"].split(",")]
    first = [(a, 1, ranks[a % len(ranks)]) for a in range(case["adapters"])]
    return first + [(a, 2, ranks[a % len(ranks)]) for a in range(min(case["versions"], case["adapters"]))]


def _popularity(case):
    """Probability of every entry, and of none (last): Zipf over adapters, a second version takes half."""
    p = np.arange(1, case["adapters"] + 1, dtype=np.float64) ** -ZIPF
    p /= p.sum()
    second = p[:min(case["versions"], case["adapters"])] / 2
    p[:len(second)] /= 2
    p = np.concatenate([p, second]) * (1 - case["none"])
    return np.concatenate([p, [case["none"]]])


def _binding(case, rng):
    """Entry per token (-1: none)."""
    p, T = _popularity(case), case["tokens"]
    none = len(p) - 1
    if case["runs"]:
        cuts = np.sort(rng.choice(np.arange(1, T), size=min(case["runs"], T) - 1, replace=False)) if T > 1 else np.array([], int)
        lengths = np.diff(np.concatenate([[0], cuts, [T]]))
        e = np.repeat(rng.choice(len(p), size=len(lengths), p=p), lengths)
    else:
        e = rng.choice(len(p), size=T, p=p)
    return np.where(e == none, -1, e).astype(np.int32)


def _segments(entry_of_token):
    cuts = np.flatnonzero(np.diff(entry_of_token)) + 1
    return (np.concatenate([[0], cuts, [len(entry_of_token)]]).astype(np.int32),
            entry_of_token[np.concatenate([[0], cuts])].astype(np.int32))


def work(case) -> dict:
    T, p, entries = case["tokens"], _popularity(case), _entries(case)
    draws = min(case["runs"], T) if case["runs"] else T
    used = 1 - (1 - p[:-1]) ** draws                                   # expected share of passes that use the entry
    rank_used = sum(u * r for u, (_, _, r) in zip(used, entries))      # rows of A (columns of B) read
    rank_tokens = T * sum(q * r for q, (_, _, r) in zip(p, entries))   # sum of ranks over the tokens
    passes = {"dual": 2, "train": 1}.get(case["kind"], 1)
    bytes_, flops, seen = 0.0, 0.0, set()
    for name, k, n, src in _sites(case):
        x_bytes = 0 if src in seen else 2 * T * k
        seen.add(src)
        weights, low = 2.0 * k * n, 2.0 * rank_used * (k + n)
        bytes_ += weights + x_bytes + low + passes * 2 * T * n
        flops += 2.0 * T * k * n + passes * 2 * rank_tokens * (k + n)
        if case["kind"] == "dual":                                     # the staged version's adapters too
            bytes_ += low / max(1, case["adapters"])
        if case["kind"] == "publish":                                  # the new version: read, and kept
            bytes_ += 2 * 2.0 * entries[0][2] * (k + n)
        if case["kind"] == "train":                                    # dx, then dA and dB in fp32
            bytes_ += weights + 2 * T * n + low + 2 * T * k + 4.0 * rank_used * (k + n)
            flops += 2.0 * T * k * n + 2 * rank_tokens * (k + n) + 2 * rank_tokens * (k + n)
    return {"bytes": bytes_, "flops": flops}


# ---- state --------------------------------------------------------------------------------------------

class _Site:
    pass


class _Inputs:
    """Everything a case draws from its seed: the binding, the activations and every site's weights and adapters."""

    def __init__(self, case, seed):
        gen = torch.Generator(device="cuda").manual_seed(int(seed))

        def normal(*shape, std=1.0):
            return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32).mul_(std).to(torch.bfloat16)

        T, entries = case["tokens"], _entries(case)
        self.entry = _binding(case, np.random.Generator(np.random.Philox(key=[int(seed), 1])))
        self.x, self.sites = {}, []
        for name, k, n, src in _sites(case):
            if src not in self.x:
                self.x[src] = normal(T, k)
            s = _Site()
            s.name, s.k, s.n, s.src = name, k, n, src
            s.W0 = normal(n, k, std=STD)
            s.A = [normal(r, k, std=STD) for _, _, r in entries]
            s.B = [normal(n, r, std=STD) for _, _, r in entries]
            if case["kind"] == "publish":
                s.new = (normal(entries[0][2], k, std=STD), normal(n, entries[0][2], std=STD))
            if case["kind"] == "train":
                s.dy = normal(T, n)
            self.sites.append(s)


def prepare(case, seed):
    """Weights, adapters registered in their tables, activations and the binding of the batch."""
    kind, T, entries, inputs = case["kind"], case["tokens"], _entries(case), _Inputs(case, seed)
    entry = inputs.entry
    ints = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).cuda()  # noqa: E731
    state = dict(case=case, sites=inputs.sites, x=inputs.x)
    for s in inputs.sites:
        s.table = Table(s.k, s.n, max_slots=len(entries) + SPARE_SLOTS)
        slots = [s.table.register_adapter(a, v, A, B, SCALE) for (a, v, _), A, B in zip(entries, s.A, s.B)]
        if kind == "publish":
            for a in range(case["adapters"]):
                s.table.publish(a, 1)
        if kind == "train":
            s.W0T = s.W0.t().contiguous()
            s.table_T = Table(s.n, s.k, max_slots=len(entries) + SPARE_SLOTS)
            s.slots_T = [s.table_T.register_adapter_transposed(a, v, A, B, SCALE) for (a, v, _), A, B in zip(entries, s.A, s.B)]
            s.dA = torch.zeros((s.table.max_slots, 64, s.k), dtype=torch.float32, device="cuda")
            s.dB = torch.zeros((s.table.max_slots, s.n, 64), dtype=torch.float32, device="cuda")
    state["version"] = 1
    # every site registered its entries in the same order, so the slot of an entry is the same everywhere
    slot_of = lambda e: np.where(e < 0, -1, np.asarray(slots, dtype=np.int32)[e])  # noqa: E731
    offsets, seg_entry = _segments(entry)
    state["slots"] = ints(slot_of(entry))
    state["adapters"] = ints(np.where(entry < 0, -1, entry))           # publish: entry e is adapter e, version 1
    state["offsets"], state["seg_slots"] = ints(offsets), ints(slot_of(seg_entry))
    # dual: the second binding has adapter 0's tokens on the entry that was resident last (the staged version)
    state["seg_slots_b"] = ints(slot_of(np.where(seg_entry == 0, len(entries) - 1, seg_entry)))
    if kind == "host":
        s = state["sites"][0]
        state["x_host"] = state["x"][0].cpu().pin_memory()
        state["y_host"] = torch.zeros((T, s.table.d_out), dtype=torch.bfloat16).pin_memory()
        state["offsets_host"] = torch.from_numpy(offsets).pin_memory()
        state["slots_host"] = torch.from_numpy(slot_of(seg_entry).astype(np.int32)).pin_memory()
    if kind == "layer":
        # the runtime keeps a workspace per group of projections and warms the layer up before it takes requests
        groups = [state["sites"][:3], state["sites"][3:4], state["sites"][4:6], state["sites"][6:]]
        state["ws"] = [torch.empty(max(256, lml_multi_workspace_bytes([s.table.handle for s in g], T)), dtype=torch.uint8, device="cuda")
                       for g in groups]
        _layer(state)
        torch.cuda.synchronize()
    if case["graph"]:
        state["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(state["graph"]):
            state["out"] = _layer(state)
    return state


# ---- one pass -----------------------------------------------------------------------------------------

def _layer(state):
    """Token-form calls over the layer's projections."""
    q, k, v, o, gate, up, down = state["sites"]
    x, slots, ws = state["x"], state["slots"], state["ws"]
    out = multi_projection([q.table, k.table, v.table], x[0], [q.W0, k.W0, v.W0], slots, workspace=ws[0])
    out.append(o.table.lora_mixed_linear_tokens(x[1], o.W0, slots, workspace=ws[1]))
    out += multi_projection([gate.table, up.table], x[2], [gate.W0, up.W0], slots, workspace=ws[2])
    out.append(down.table.lora_mixed_linear_tokens(x[3], down.W0, slots, workspace=ws[3]))
    return out


def run(state):
    case, x = state["case"], state["x"]
    kind = case["kind"]
    if kind == "layer":
        if case["graph"]:
            state["graph"].replay()
            return state["out"]
        return _layer(state)
    if kind in ("segments", "small"):
        return [s.table.lora_mixed_linear(x[s.src], s.W0, state["offsets"], state["seg_slots"]) for s in state["sites"]]
    if kind == "publish":
        state["version"] += 1
        for s in state["sites"]:
            s.table.register_adapter(0, state["version"], s.new[0], s.new[1], SCALE)
            s.table.publish(0, state["version"])
        return [s.table.lora_mixed_linear_adapters(x[s.src], s.W0, state["adapters"]) for s in state["sites"]]
    if kind == "dual":
        return [s.table.lora_mixed_linear_dual(x[s.src], s.W0, state["offsets"], state["seg_slots"], state["seg_slots_b"])
                for s in state["sites"]]
    if kind == "train":
        out = [s.table.lora_mixed_linear(x[s.src], s.W0, state["offsets"], state["seg_slots"]) for s in state["sites"]]
        for s in reversed(state["sites"]):
            # transposed tables were filled in the same order: slots are the same in both
            out.append(s.table_T.lora_mixed_linear(s.dy, s.W0T, state["offsets"], state["seg_slots"]))
            s.dA.zero_()
            s.dB.zero_()
            s.table.backward_adapters(s.table_T, x[s.src], s.dy, state["offsets"], state["seg_slots"], state["seg_slots"], s.dA, s.dB)
            out += [s.dA, s.dB]
        return out
    s = state["sites"][0]
    s.table.lora_mixed_linear_host(state["x_host"], s.W0, state["offsets_host"], state["slots_host"], state["y_host"])
    torch.cuda.current_stream().synchronize()                          # y_host is valid from here on: the caller reads it
    return state["y_host"]


def tolerance(case) -> dict:
    # y is bf16 and rounded once, and u is rounded to bf16 before the expand on some paths: against a float64 evaluation y is off
    # by rel 1.7e-3 and max 6e-3 at most.  dA and dB are float32 sums of products with bf16-rounded u: rel 1.8e-3, but an element
    # near zero is a sum that cancels, so its error is up to 0.037 of the matrix's root mean square.
    return {"rel": 7e-3, "max": 0.15} if case["kind"] == "train" else {"rel": 7e-3, "max": 0.025}


def exact(case, seed):
    """What run() returns for these inputs, in 64 bits: entry e is in slot e (the first registrations of an empty table)."""
    inputs, entries, kind = _Inputs(case, seed), _entries(case), case["kind"]
    wide = lambda t: t.to(torch.float64)  # noqa: E731

    def rows(entry, e):
        return torch.from_numpy(np.flatnonzero(entry == e)).cuda()

    def layer(x, W, A, B, entry):
        x = wide(x)
        y = x @ wide(W).t()
        for e in range(len(A)):
            at = rows(entry, e)
            y[at] += SCALE * ((x[at] @ wide(A[e]).t()) @ wide(B[e]).t())
        return y

    out = []
    for s in inputs.sites:
        x, A = inputs.x[s.src], list(s.A)
        B = list(s.B)
        if kind == "publish":
            A[0], B[0] = s.new
        y = layer(x, s.W0, A, B, inputs.entry)
        if kind == "dual":
            y = (y, layer(x, s.W0, A, B, np.where(inputs.entry == 0, len(entries) - 1, inputs.entry)))
        out.append(y)
    if kind == "host":
        return out[0].cpu()
    if kind == "train":
        for s in reversed(inputs.sites):
            x, dy = wide(inputs.x[s.src]), wide(s.dy)
            out.append(layer(s.dy, s.W0.t(), [B.t() for B in s.B], [A.t() for A in s.A], inputs.entry))
            dA = torch.zeros((len(entries) + SPARE_SLOTS, 64, s.k), dtype=torch.float64, device="cuda")
            dB = torch.zeros((len(entries) + SPARE_SLOTS, s.n, 64), dtype=torch.float64, device="cuda")
            for e, (_, _, r) in enumerate(entries):
                at = rows(inputs.entry, e)
                dA[e, :r] = SCALE * ((dy[at] @ wide(s.B[e])).t() @ x[at])
                dB[e, :, :r] = SCALE * (dy[at].t() @ (x[at] @ wide(s.A[e]).t()))
            out += [dA, dB]
    return out
