"""Performance cases of the decode hot path: what a serving program has the library do, through its public calls.

Two kinds of case.

`attend`   one query token over a caller-owned K/V buffer (`wnw_attend_static`).

`request`  what a server does with a batch of requests on a cache that it keeps: place the prefill K,V of every sequence,
           layer by layer, then decode `steps` tokens, each through all layers with its K,V row appended to the text.  The
           tokens are decoded by replaying a captured step (`issue` = graph: the step is captured once per placed batch,
           as the library asks for) or call by call (`issue` = eager).  A pass starts with the placement, so it can be
           repeated on the same cache; few steps measure the way to the first token, many steps measure decoding.

The numbers of a case: model shape (layers, q_heads, kv_heads, dim), batch, audio tokens per sequence (`ragged`: uniform
between a quarter of that and that), text prefix, chunk, budget, steps, and the options a program chooses (how layers depend
on one another, storage format of the tidal tier, residency, token-granular compression, text queries that rank the
prefill, audio arriving while tokens are decoded, full-cache storage).

Inputs follow the structure that attention over speech shows: a sink on the first audio positions, and a decode focus that
drifts through the clip once per `sweep` steps (`sweep` = 0: jumps every four steps), so that chunks go out of and come back
into the GPU's slots at the rate they do in decoding.
"""
import math

import numpy as np
import torch

from paper_2608_22704_b200 import binding as wnw

REGION = 64      # audio tokens that share one direction in the synthetic keys

DEPENDENCY = {"chained": wnw.WNW_LAYERS_CHAINED, "independent": wnw.WNW_LAYERS_INDEPENDENT, "batched": wnw.WNW_LAYERS_BATCHED}


def _request(name=None, **changes):
    case = dict(kind="request", layers=30, q_heads=32, kv_heads=8, dim=128, batch=1, audio=3000, ragged=False, text=64, chunk=64,
                budget=0.2, steps=64, sweep=256, issue="graph", layer_order="chained", storage="bf16", segments=False, tokens=False,
                queries=1, append=0, full=False)
    case.update(changes)
    if name:
        case["name"] = name
    return case


def listed():
    return [
        # the smallest call: one token of a small model over half a minute of audio, in a loop that must not allocate
        dict(name="attend_short", kind="attend", q_heads=8, kv_heads=4, dim=64, tokens=777),
        # one token of a 3B model over an hour-long context
        dict(name="attend_long", kind="attend", q_heads=32, kv_heads=8, dim=128, tokens=50001),
        # a single small layer driven call by call: launch and host latency
        _request("tiny_eager", layers=1, q_heads=8, kv_heads=4, dim=64, audio=1024, text=32, chunk=32, steps=16, sweep=16, issue="eager"),
        # 3B model, four minutes of audio: the way from the prefill K,V to the first token
        _request("first_token", steps=1, issue="eager"),
        # the same request decoded to its end by a decoder whose layers feed one another: the everyday case
        _request("decode_4min", steps=256),
        # ten minutes of audio at the higher frame rate, few KV heads: long heads, large groups
        _request("decode_10min", layers=36, q_heads=16, kv_heads=2, audio=15000, steps=128, sweep=512),
        # several requests, all queries of a step known ahead (layers need not wait for one another)
        _request("decode_independent", batch=4, steps=96, layer_order="independent"),
        # batched serving of clips of different lengths
        _request("batch_ragged", layers=6, batch=16, audio=7500, ragged=True, steps=128, sweep=128),
        # recall-bound serving: the focus jumps, the tidal tier is stored as e4m3 to halve the link's bytes
        _request("batch_recall_e4m3", layers=4, batch=16, audio=7500, steps=64, sweep=0, storage="e4m3"),
        # the paper's own form: segments of two seconds, a token-granular base, every head's retention its own, text queries
        _request("paper_form", layers=30, chunk=25, segments=True, tokens=True, queries=4, steps=64, sweep=1200),
        # streaming: two seconds of audio arrive, a few tokens are decoded, and so on; an open-ended loop, so call by call
        _request("streaming", layers=30, audio=1487, steps=24, issue="eager", append=25, sweep=48),
        # the full-cache baseline of the same model
        _request("full_cache", batch=4, steps=64, full=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    limit = [_load(c) for c in listed()]
    limit = [max(x) for x in zip(*limit)]
    while True:
        case = _draw(rng)
        if all(x <= y for x, y in zip(_load(case), limit)):
            return case


def _draw(rng):
    q_heads, kv_heads, dim = rng.choice([(8, 4, 64), (32, 8, 128), (32, 8, 128), (16, 2, 128), (16, 4, 64)])
    if rng.random() < 0.2:
        return dict(kind="attend", q_heads=q_heads, kv_heads=kv_heads, dim=dim, tokens=_log_int(rng, 300, 80000))
    form = rng.choice(["single", "single", "batch", "batch", "e4m3", "paper", "streaming", "full"])
    case = _request(q_heads=q_heads, kv_heads=kv_heads, dim=dim, layers=_log_int(rng, 1, 36), audio=_log_int(rng, 700, 15000),
                    text=_log_int(rng, 16, 200), chunk=rng.choice([32, 50, 64, 64, 100, 128]), budget=rng.choice([0.1, 0.2, 0.2, 0.3]),
                    steps=_log_int(rng, 1, 256), sweep=rng.choice([0, 128, 256, 512, 1200]),
                    issue=rng.choice(["graph", "graph", "eager"]), layer_order=rng.choice(["chained", "chained", "independent", "batched"]))
    if form in ("batch", "e4m3", "full"):
        case.update(batch=_log_int(rng, 2, 24), audio=_log_int(rng, 1000, 7500), ragged=rng.random() < 0.5)
    if form == "e4m3":
        case.update(storage="e4m3", q_heads=32, kv_heads=8, dim=128)
    elif form == "paper":
        case.update(chunk=rng.choice([25, 50]), segments=True, tokens=True, queries=rng.randint(1, 6), audio=_log_int(rng, 1000, 6000))
    elif form == "streaming":
        case.update(append=rng.randint(5, 60), issue="eager", steps=4 * rng.randint(1, 8), sweep=64)
    elif form == "full":
        case.update(full=True)
    return case


def _load(case):
    """What bounds a case's cost: bytes, layer launches of the decode loop, placements, bytes of the prefill."""
    if case["kind"] == "attend":
        return work(case)["bytes"], 0, 0, 0
    tokens = sum(_lengths(case)) + case["batch"] * case["text"]
    return (work(case)["bytes"], case["steps"] * case["layers"] * (4 if case["issue"] == "eager" else 1), case["layers"] * case["batch"],
            tokens * case["layers"] * case["kv_heads"] * case["dim"] * 4 * case["queries"])


# ---------------------------------------------------------------------------------------------------------------- shapes
def _lengths(case):
    if not case["ragged"]:
        return [case["audio"]] * case["batch"]
    rs = np.random.RandomState(case["batch"] * 8191 + case["audio"])
    return [int(x) for x in rs.randint(case["audio"] // 4, case["audio"] + 1, case["batch"])]


def _roles(case):
    """Offline head roles of the model: one head in eight an anchor (at least one a layer), a quarter fixed, the rest tidal;
    with two KV heads a layer, drawn per layer and an anchor in every fourth layer at least."""
    L, H = case["layers"], case["kv_heads"]
    rs = np.random.RandomState(1000 * H + L)
    A, T, F = wnw.WNW_ROLE_ANCHOR, wnw.WNW_ROLE_TIDAL, wnw.WNW_ROLE_FIXED
    if H >= 4:
        base = np.array([A] * max(1, H // 8) + [F] * (H // 4), np.uint8)
        base = np.concatenate([base, np.full(H - len(base), T, np.uint8)])
        return np.stack([base[rs.permutation(H)] for _ in range(L)])
    u = rs.random_sample((L, H))
    roles = np.where(u < 1 / 8, A, np.where(u < 5 / 8, T, F)).astype(np.uint8)
    for first in range(0, L, 4):
        block = roles[first:first + 4]
        if not (block == A).any():
            block[rs.randint(0, len(block)), rs.randint(0, H)] = A
    return roles


def _retention(case):
    """Per-head retention around the budget (Eq. 1 gives a head its own)."""
    rs = np.random.RandomState(7 + case["layers"])
    return (case["budget"] * (0.75 + 0.5 * rs.random_sample((case["layers"], case["kv_heads"])))).astype(np.float32)


def _appended_before(case, step):
    """Audio positions that have arrived before a decode step: one arrival ahead of every fourth step."""
    return case["append"] * (step // 4 + 1) if case["append"] else 0


# ---------------------------------------------------------------------------------------------------------------- inputs
class _State:
    """Inputs and the handle of a case; the cache goes with it."""

    def __init__(self):
        self.cache = None

    def __del__(self):
        if self.cache is not None:
            wnw.wnw_destroy(self.cache)


def prepare(case, seed):
    s = _State()
    s.case = case
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)

    def randn(*shape, dtype=torch.bfloat16):
        return torch.randn(*shape, generator=gen, device="cuda", dtype=dtype)

    Hq, H, d = case["q_heads"], case["kv_heads"], case["dim"]
    if case["kind"] == "attend":
        n = case["tokens"]
        s.kv = randn(H, 2, (n + 15) // 16 * 16, d)
        s.q = randn(Hq, d) * 2
        s.out = torch.empty(Hq, d, dtype=torch.bfloat16, device="cuda")
        return s

    L, B, N, n_text = case["layers"], case["batch"], case["steps"], case["text"]
    lengths = _lengths(case)
    grown = [a + _appended_before(case, N - 1) for a in lengths]
    group = Hq // H
    s.lengths = lengths
    s.prefill = []                                      # per sequence: K, V [L][tokens][H][d], text queries [L][queries][Hq][d]
    s.arriving = []                                     # per sequence: K, V [arrivals][L][append][H][d]
    s.q = torch.empty(N, L, B, Hq, d, dtype=torch.bfloat16, device="cuda")
    for b, T_a in enumerate(lengths):
        sink = torch.nn.functional.normalize(randn(L, H, d, dtype=torch.float32), dim=-1)
        codes = torch.nn.functional.normalize(randn(L, H, -(-grown[b] // REGION), d, dtype=torch.float32), dim=-1)
        k, v = randn(L, n_text + T_a, H, d), randn(L, n_text + T_a, H, d)
        code_rows = (4.0 * codes).to(torch.bfloat16).transpose(1, 2)            # [L][regions][H][d]
        region = torch.arange(grown[b], device="cuda") // REGION
        k[:, n_text:] += code_rows[:, region[:T_a]]
        k[:, n_text:n_text + 4] += (4.0 * sink).to(torch.bfloat16).unsqueeze(1)
        lean = sink.repeat_interleave(group, dim=1).unsqueeze(1)                # [L][1][Hq][d]
        q_text = randn(L, case["queries"], Hq, d, dtype=torch.float32) + 2.0 * math.sqrt(d) * lean
        s.prefill.append((k, v, q_text.to(torch.bfloat16)))
        if case["append"]:
            n_new = grown[b] - T_a
            ka, va = randn(L, n_new, H, d) + code_rows[:, region[T_a:]], randn(L, n_new, H, d)
            split = lambda x: x.view(L, -1, case["append"], H, d).transpose(0, 1).contiguous()  # noqa: E731
            s.arriving.append((split(ka), split(va)))
        # the decode focus: a bell over regions around its centre
        t = torch.arange(N, device="cuda", dtype=torch.float32)
        if case["sweep"]:
            centre = (t / case["sweep"]) % 1.0
        else:
            centre = torch.rand(-(-N // 4), generator=gen, device="cuda").repeat_interleave(4)[:N]
        centre = centre * grown[b] / REGION
        r = torch.arange(codes.shape[2], device="cuda", dtype=torch.float32)
        bell = torch.exp(-0.5 * (r + 0.5 - centre.unsqueeze(1)) ** 2)           # [N][regions]
        focus = torch.einsum("tr,lhrd->tlhd", bell, codes)
        bias = math.sqrt(d) * (0.5 * sink.unsqueeze(0) + 1.5 * focus)
        s.q[:, :, b] = (randn(N, L, Hq, d, dtype=torch.float32) + bias.repeat_interleave(group, dim=2)).to(torch.bfloat16)
    s.k_new, s.v_new = randn(N, L, B, H, d), randn(N, L, B, H, d)
    s.out = torch.zeros(N, L, B, Hq, d, dtype=torch.bfloat16, device="cuda")
    s.retention = _retention(case)
    s.cache = wnw.wnw_create(
        L, Hq, H, d, B, max(grown), n_text + N, case["chunk"], case["budget"], _roles(case),
        mode=wnw.WNW_MODE_FULL if case["full"] else wnw.WNW_MODE_TIERED,
        residency=(wnw.WNW_RESIDENCY_HARD_BUDGET if not case["segments"] else
                   wnw.WNW_RESIDENCY_SEGMENT_LAG_TOKEN_BASE if case["tokens"] else wnw.WNW_RESIDENCY_SEGMENT_LAG),
        score_scope=wnw.WNW_SCOPE_GLOBAL if case["segments"] else wnw.WNW_SCOPE_PER_LAYER,
        streaming_audio=1 if case["append"] else 0,
        tidal_kv_format=wnw.WNW_TIDAL_KV_FP8_E4M3 if case["storage"] == "e4m3" else wnw.WNW_TIDAL_KV_BF16)
    wnw.wnw_set_layer_dependency(s.cache, DEPENDENCY[case["layer_order"]])
    s.stream = torch.cuda.Stream()
    if case["issue"] == "graph":      # the buffers a captured step reads and writes: q, k_new, v_new of one step, and its outputs
        s.step_q, s.step_k, s.step_v, s.step_out = (torch.zeros_like(x[0]) for x in (s.q, s.k_new, s.v_new, s.out))
    return s


# ---------------------------------------------------------------------------------------------------------------- passes
def run(s):
    if s.case["kind"] == "attend":
        wnw.wnw_attend_static(s.kv, s.case["tokens"], s.q, s.out)
        return s.out
    s.stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s.stream):
        _place(s)
        (_decode_graph if s.case["issue"] == "graph" else _decode_eager)(s)
    torch.cuda.current_stream().wait_stream(s.stream)
    return s.out


def _place(s):
    case, begin = s.case, s.case["text"]
    for b, (k, v, q_text) in enumerate(s.prefill):
        end = begin + s.lengths[b]
        for layer in range(case["layers"]):
            q = q_text[layer] if case["queries"] > 1 or case["tokens"] else q_text[layer, 0]
            if case["tokens"]:
                wnw.wnw_place_prefill_tokens(s.cache, b, layer, k[layer], v[layer], begin, end, q, s.retention[layer], case["chunk"],
                                             stream=s.stream)
            else:
                wnw.wnw_place_prefill(s.cache, b, layer, k[layer], v[layer], begin, end, q, stream=s.stream)


def _step(s, q, k_new, v_new, out):
    layer_call = wnw.wnw_decode_layer_full if s.case["full"] else wnw.wnw_decode_layer
    wnw.wnw_step_begin(s.cache, range(s.case["batch"]))
    for layer in range(s.case["layers"]):
        layer_call(s.cache, layer, q[layer], k_new[layer], v_new[layer], out[layer], stream=s.stream)
    wnw.wnw_step_end(s.cache, stream=s.stream)


def _decode_eager(s):
    for t in range(s.case["steps"]):
        if s.case["append"] and t % 4 == 0:
            for b, (k, v) in enumerate(s.arriving):
                for layer in range(s.case["layers"]):
                    wnw.wnw_append_audio(s.cache, b, layer, k[t // 4, layer], v[t // 4, layer], stream=s.stream)
        _step(s, s.q[t], s.k_new[t], s.v_new[t], s.out[t])


def _decode_graph(s):
    wnw.wnw_graph_begin(s.cache, range(s.case["batch"]), s.stream)
    _step(s, s.step_q, s.step_k, s.step_v, s.step_out)
    wnw.wnw_graph_end(s.cache, s.stream)
    for t in range(s.case["steps"]):
        s.step_q.copy_(s.q[t])
        s.step_k.copy_(s.k_new[t])
        s.step_v.copy_(s.v_new[t])
        wnw.wnw_graph_launch(s.cache, s.stream)
        s.out[t].copy_(s.step_out)


# ---------------------------------------------------------------------------------------------------------------- floors
def work(case):
    """Bytes: every input and output once, every K,V row that a token attends to once per token, and the placed tiers written
    once.  Recalled chunks are not counted (how many there are depends on the queries)."""
    Hq, H, d = case["q_heads"], case["kv_heads"], case["dim"]
    if case["kind"] == "attend":
        return {"bytes": 4 * d * H * case["tokens"] + 4 * Hq * d, "flops": 4 * Hq * d * case["tokens"]}
    L, N, group = case["layers"], case["steps"], Hq // H
    roles = _roles(case)
    n_role = [int((roles == r).sum()) for r in (wnw.WNW_ROLE_ANCHOR, wnw.WNW_ROLE_TIDAL, wnw.WNW_ROLE_FIXED)]
    if case["full"]:
        n_role = [L * H, 0, 0]
    tidal_row = 2 * d if case["storage"] == "e4m3" else 4 * d
    total, flops = 0.0, 0.0
    for T_a in _lengths(case):
        prefix = case["text"] + T_a
        kept = max(1.0, case["budget"] * T_a)
        total += 4 * d * L * H * prefix + 2 * d * L * Hq * case["queries"]                                     # inputs
        total += 4 * d * (L * H * case["text"] + n_role[0] * T_a + n_role[2] * kept) + tidal_row * n_role[1] * (T_a + kept)
        if not case["full"]:
            flops += 2 * Hq * d * L * prefix * case["queries"]
        for t in range(N):
            text, audio = case["text"] + t + 1, T_a + _appended_before(case, t)
            total += 4 * d * (L * H * text + n_role[0] * audio + n_role[2] * kept) + tidal_row * n_role[1] * kept
            flops += 4 * d * group * (L * H * text + n_role[0] * audio + (n_role[1] + n_role[2]) * kept)
        total += N * L * 2 * d * (2 * Hq + 4 * H)                                        # queries, outputs, new rows read and stored
        total += 8 * d * L * H * _appended_before(case, N - 1)                           # audio that arrives while decoding
    return {"bytes": total, "flops": flops}


def tolerance(case):
    # bf16 outputs of fp32 sums over bf16 products; softmax weights rounded to bf16 against a maximum that depends on the split
    return {"rel": 1e-2, "max": 0.2}
