"""The calls a serving engine makes on this library, as cases that can be timed and compared.

A prefix cache stores a checkpoint of the recurrent states (``dasc_pack``, ``dasc_pack_int8``), loads it again on a hit
(``dasc_restore``, ``dasc_restore_int8``) and replays the tokens behind the checkpoint (``dasc_refresh``) or the last
tokens before it (``dasc_refresh_window``).  Shapes are those of the benchmark configurations: 24 KDA layers of 32 heads
or 36 GDN layers of 32 value / 16 key heads, d_k = d_v = 128, fp32 states, a rank of a tensor-parallel group holding
fewer heads; a store or a load moves all layers of a checkpoint, a refresh call covers one layer (a forward pass goes
layer by layer) or a group of layers.
"""
import math

import torch

import paper_2608_30386_b200 as dasc
from paper_2608_30386_b200 import synth

DEVICE = "cuda"
RATE_LO = {"KDA": 1e-3, "GDN": 1e-4}  # decay rates are log-uniform from here to 1
MOST_BYTES = 7.2e9                    # what the largest listed copy moves
MOST_TOKEN_HEADS = 2.1e6              # what the largest listed refresh replays


def _copy(op, pool, kind, layers, v_heads, requests, keep):
    return {"op": op, "pool": pool, "kind": kind, "layers": layers, "v_heads": v_heads,
            "k_heads": v_heads if kind == "KDA" else v_heads // 2, "dim": 128, "requests": requests, "keep": keep}


def _refresh(kind, layers, v_heads, requests, tokens, ragged, streams="bf16", dim=128, keep=0.38, window=0):
    return {"op": "window" if window else "refresh", "kind": kind, "layers": layers, "v_heads": v_heads,
            "k_heads": v_heads if kind == "KDA" else v_heads // 2, "dim": dim, "requests": requests, "keep": keep,
            "tokens": tokens, "ragged": ragged, "streams": streams, "window": window}


def listed():
    return [
        # a request reaches a checkpoint boundary on its own; a single hit is loaded
        {"name": "store_one", **_copy("store", "fp32", "KDA", 24, 32, 1, 0.38)},
        {"name": "load_one", **_copy("load", "fp32", "KDA", 24, 32, 1, 0.38)},
        # a whole batch at once: the serving-scale KDA configuration, the head-wise GDN configuration
        {"name": "store_batch", **_copy("store", "fp32", "KDA", 24, 32, 64, 0.38)},
        {"name": "load_batch_gdn", **_copy("load", "fp32", "GDN", 36, 32, 64, 0.5)},
        # the same with the INT8 checkpoint pool, a batch size that is no power of two
        {"name": "store_int8", **_copy("store", "int8", "KDA", 24, 32, 37, 0.38)},
        {"name": "load_int8", **_copy("load", "int8", "KDA", 24, 32, 37, 0.38)},
        # suffix refresh of a batch over a group of layers, both kinds
        {"name": "refresh_kda", **_refresh("KDA", 4, 32, 64, 256, False)},
        {"name": "refresh_gdn", **_refresh("GDN", 4, 32, 64, 256, False, keep=0.5)},
        # mixed serving trace: hits with 1 .. 1023 tokens since their checkpoint, one layer of the forward pass
        {"name": "refresh_ragged_layer", **_refresh("KDA", 1, 32, 64, 512, True)},
        # one hit alone, one layer: latency
        {"name": "refresh_one", **_refresh("KDA", 1, 32, 1, 509, False)},
        # load policy that replays the last tokens of the prefix from a zero state; no outputs
        {"name": "window_kda", **_refresh("KDA", 4, 32, 32, 256, True, window=128)},
        # the tiny fp32 configuration
        {"name": "refresh_fp32_tiny", **_refresh("KDA", 1, 4, 1, 64, False, streams="fp32", dim=64, keep=0.4)},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["KDA", "KDA", "GDN"])
    heads = rng.choice([4, 8, 16, 32, 32])
    keep = rng.choice([0.2, 0.25, 0.38, 0.5])
    if rng.random() < 0.4:
        case = _copy(rng.choice(["store", "load"]), rng.choice(["fp32", "int8"]), kind, 24 if kind == "KDA" else 36, heads,
                     _log_uniform(rng, 1, 64), keep)
        while work(case)["bytes"] > MOST_BYTES:
            case["requests"] -= 1
        return case
    if rng.random() < 0.2:  # fp32 streams: small models and checks
        dim = rng.choice([64, 128])
        case = _refresh(kind, rng.choice([1, 2]), rng.choice([4, 8]), _log_uniform(rng, 1, 16), _log_uniform(rng, 16, 256),
                        rng.random() < 0.5, streams="fp32", dim=dim, keep=keep)
    else:
        window = rng.choice([16, 64, 128, 512]) if rng.random() < 0.25 else 0
        tokens = 2 * window if window else _log_uniform(rng, 5, 4096)
        case = _refresh(kind, rng.choice([1, 1, 2, 4]), heads, _log_uniform(rng, 1, 64), tokens, rng.random() < 0.6, keep=keep,
                        window=window)
    per_request = case["layers"] * case["v_heads"] * case["tokens"]
    case["requests"] = max(1, min(case["requests"], int(MOST_TOKEN_HEADS // per_request)))
    return case


def _plan(case, gen):
    per_head = case["dim"] if case["kind"] == "KDA" else 1
    rates = synth.decay_rates(gen, case["layers"], case["v_heads"], per_head, RATE_LO[case["kind"]], 1.0)
    a_log, dt_bias = synth.decay_params(rates)
    plan = dasc.dasc_plan(dasc.KDA if case["kind"] == "KDA" else dasc.GDN, case["layers"], case["v_heads"], case["k_heads"],
                          case["dim"], case["dim"], a_log, dt_bias, sel=dasc.SEL_TOP_RATIO, scope=dasc.SCOPE_LAYER,
                          keep_ratio=case["keep"], device=torch.cuda.current_device())
    return plan, rates


def _lengths(case, gen):
    """Tokens of each request: `tokens` each, or spread over 1 .. 2*tokens-1 with the same total."""
    n, mean = case["requests"], case["tokens"]
    if not case["ragged"] or n == 1 or mean == 1:
        return torch.full((n,), mean, dtype=torch.int64)
    lens = torch.randint(1, 2 * mean, (n,), generator=gen, dtype=torch.int64)
    i, excess = 0, int(lens.sum()) - n * mean
    while excess:  # even out the total, a request at a time
        new = min(max(int(lens[i]) - excess, 1), 2 * mean - 1)
        excess -= int(lens[i]) - new
        lens[i] = new
        i += 1
    return lens


def prepare(case, seed):
    host, dev = synth.generator(seed), synth.generator(seed, DEVICE)
    plan, rates = _plan(case, host)
    n, layers, dense = case["requests"], case["layers"], case["v_heads"] * case["dim"] ** 2
    ids = torch.arange(n, dtype=torch.int32, device=DEVICE)
    s = {"case": case, "plan": plan, "ids": ids, "layer_stride": n * dense, "req_stride": dense,  # [layer][request][...]
         "state": synth.states(dev, (layers, n, dense), DEVICE)}
    if case["op"] in ("store", "load"):
        slots = n + max(1, n // 4)  # the pool is larger than the batch
        s["slot"] = torch.randperm(slots, generator=host)[:n].to(torch.int32).to(DEVICE)
        if case["pool"] == "int8":
            s["pool"] = torch.zeros((slots, dasc.dasc_int8_slot_bytes(plan)), dtype=torch.uint8, device=DEVICE)
        else:
            s["pool"] = torch.zeros((slots, int(plan.slot_floats)), device=DEVICE)
        if case["op"] == "load":  # what an earlier store left
            _store(s)
            s["state"] = torch.empty_like(s["state"])
        return s
    lens = _lengths(case, host)
    cu = torch.zeros(n + 1, dtype=torch.int64)
    cu[1:] = torch.cumsum(lens, 0)
    total = int(cu[-1])
    io = torch.bfloat16 if case["streams"] == "bf16" else torch.float32
    parts = [synth.token_streams(dev, synth.KDA if case["kind"] == "KDA" else synth.GDN, 1, total, case["v_heads"],
                                 case["k_heads"], case["dim"], case["dim"], rates[i:i + 1], io, DEVICE) for i in range(layers)]
    for f in ("q", "k", "v", "g", "beta"):
        s[f] = torch.cat([getattr(p, f) for p in parts])
    bytes_ws = dasc.dasc_refresh_workspace_bytes(plan, n, layers)
    s.update(cu=cu.to(torch.int32).to(DEVICE), total=total, longest=int(lens.max()),
             workspace=torch.zeros(max(bytes_ws, 256), dtype=torch.uint8, device=DEVICE))
    if case["op"] == "window":
        s["window_begin"] = torch.empty(n, dtype=torch.int32, device=DEVICE)
    else:
        s["o"] = torch.empty((layers, total, case["v_heads"], case["dim"]), dtype=io, device=DEVICE)
    return s


def _store(s):
    call = dasc.dasc_pack_int8 if s["case"]["pool"] == "int8" else dasc.dasc_pack
    call(s["plan"], s["state"], s["layer_stride"], s["req_stride"], s["ids"], s["pool"], s["slot"])
    return s["pool"]


def _load(s):
    call = dasc.dasc_restore_int8 if s["case"]["pool"] == "int8" else dasc.dasc_restore
    call(s["plan"], s["pool"], s["slot"], s["state"], s["layer_stride"], s["req_stride"], s["ids"])
    return s["state"]


def run(s):
    op = s["case"]["op"]
    if op == "store":
        return _store(s)
    if op == "load":
        return _load(s)
    if op == "window":
        dasc.dasc_refresh_window(s["plan"], s["state"], s["layer_stride"], s["req_stride"], s["ids"], None, s["k"], s["v"],
                                 s["g"], s["beta"], s["cu"], s["total"], s["window_begin"], window=s["case"]["window"],
                                 workspace=s["workspace"])
        return {"state": s["state"], "window_begin": s["window_begin"]}
    dasc.dasc_refresh(s["plan"], s["state"], s["layer_stride"], s["req_stride"], s["ids"], s["q"], s["k"], s["v"], s["g"],
                      s["beta"], s["cu"], s["total"], s["longest"], o=s["o"], workspace=s["workspace"])
    return {"state": s["state"], "o": s["o"]}


def work(case):
    d, kda = case["dim"], case["kind"] == "KDA"
    units = case["layers"] * case["v_heads"] * (d if kda else 1)
    kept = case["layers"] * math.ceil(case["keep"] * case["v_heads"] * (d if kda else 1) - 1e-9) / units
    rows = case["requests"] * case["layers"] * case["v_heads"] * d  # rows of d values: the codec scales each by one fp32
    dense = rows * d * 4
    if case["op"] in ("store", "load"):
        pool = kept * (rows * (d + 4) if case["pool"] == "int8" else dense)
        return {"bytes": pool + (kept * dense if case["op"] == "store" else dense), "flops": 0}
    replayed = case["tokens"]
    if case["op"] == "window":  # prefixes are spread over 1 .. 2*tokens-1: a shorter one than the window is replayed whole
        w, most = case["window"], 2 * case["tokens"] - 1
        short = min(w, most)
        replayed = (short * (short + 1) / 2 + (most - short) * w) / most if case["ragged"] and case["requests"] > 1 else min(
            w, case["tokens"])
    token_heads = case["requests"] * case["layers"] * case["v_heads"] * replayed
    io = 2 if case["streams"] == "bf16" else 4
    shared = case["k_heads"] / case["v_heads"]
    per = d * io * shared + d * io + (d * 4 if kda else 4) + 4  # k, v, g, beta
    if case["op"] == "window":  # the omitted units are written, no outputs
        return {"bytes": token_heads * per + (1 - kept) * dense, "flops": token_heads * 5 * d * d}
    return {"bytes": token_heads * (per + d * io * shared + d * io) + 2 * dense, "flops": token_heads * 7 * d * d}


def tolerance(case):
    if case["op"] in ("store", "load"):
        return "exact"  # bit copies; codes and scales of the INT8 pool are decided in fp32
    # fp32 streams are replayed in fp32; bf16 streams with tf32 products, and their outputs are rounded to bf16
    return {"rel": 1e-5} if case["streams"] == "fp32" else {"rel": 2e-3}
