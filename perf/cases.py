"""The calls whose speed is tracked, from the smallest to the largest that a user of the library makes.

A user of this library is a multi-camera vision-language pipeline: per batch of requests it makes the first layer's
queries and keys (`project`), scores the visual tokens by the text's attention and keeps the best ones
(`score_topk`, `score`, `score_full_keys`, `topk`), and gathers the kept rows for the language model (`compact`,
`splice`). Every case goes through `paper_2506_07416_gb300.select`: the `Selector` object, or the functions of the
module with buffers that a server keeps. Sizes are those of this repository's workloads (camera views of 256, 576 or
1024 visual tokens, 16..128 text tokens, 14/2 to 32/32 heads of 64 or 128), and around them.

A case's request lengths are drawn from its own `sizes` number, so that a case is a dict of plain values.
"""
import math
import random

import numpy as np
import torch

from paper_2506_07416_gb300 import select

# The largest batch: 128 requests x (3456 visual + 64 text tokens), 32 heads x 128.
# Drawn batches stay well below it.
_MOST_BYTES = 2.5e9
_MOST_LOGITS = 128 * 3456 * 64 * 32 // 2    # (text row, head, visual token) triples
_MOST_PROJECT = 27648 * 4096 * 4096         # multiplications of a projection


# ------------------------------------------------------------------------------------------------------------ cases
def listed():
    return [
        # one camera view of one vehicle on a small model: nothing but latency (launches, first accesses, host path)
        dict(name="step_one_view", kind="step", batch=1, n_lo=256, n_hi=256, t_lo=32, t_hi=32, sizes=1, hq=14, hkv=2,
             d=64, hidden=896, dtype="bf16", ratio=0.5, gather="hidden"),
        # six views of one vehicle: the ordinary single-request frame
        dict(name="step_frame", kind="step", batch=1, n_lo=1536, n_hi=1536, t_lo=64, t_hi=64, sizes=2, hq=16, hkv=16,
             d=128, hidden=2048, dtype="bf16", ratio=0.3, gather="hidden"),
        # six high-resolution views, long prompt, grouped heads; K and V rows feed the cache
        dict(name="step_highres", kind="step", batch=1, n_lo=6144, n_hi=6144, t_lo=128, t_hi=128, sizes=3, hq=28,
             hkv=4, d=128, hidden=3584, dtype="bf16", ratio=0.25, gather="hidden+kv"),
        # a small serving batch of requests with odd lengths, at the paper's ratio for half-precision inputs
        dict(name="step_ragged", kind="step", batch=12, n_lo=241, n_hi=3089, t_lo=19, t_hi=127, sizes=4, hq=32, hkv=8,
             d=128, hidden=4096, dtype="bf16", ratio=0.8, gather="hidden+kv"),
        # an 8-bit serving batch, 1..6 views a request, a count of its own to keep, buffers kept by the server
        dict(name="step_fp8_ragged", kind="step_buffers", batch=32, n_lo=576, n_hi=3456, t_lo=32, t_hi=128, sizes=5,
             hq=32, hkv=32, d=128, hidden=4096, dtype="e4m3", ratio=0.2, gather="hidden"),
        # the largest batch: scores of 128 requests of six views
        dict(name="score_sweep", kind="score", batch=128, n_lo=3456, n_hi=3456, t_lo=64, t_hi=64, sizes=6, hq=32,
             hkv=32, d=128, hidden=4096, dtype="bf16", ratio=0.3, gather="hidden", query="all"),
        # the other half of a large batch: top-k of its scores and the spliced prefill input
        dict(name="prefill_batch", kind="prefill", batch=64, n_lo=2900, n_hi=3500, t_lo=33, t_hi=127, sizes=7, hq=32,
             hkv=32, d=128, hidden=4096, dtype="bf16", ratio=0.3, gather="hidden", s_lo=17, s_hi=48),
        # scores whose softmax runs over the whole causal prompt (system, image, text), ragged, with a top-k after it
        dict(name="full_keys_ragged", kind="full_keys", batch=16, n_lo=512, n_hi=3072, t_lo=24, t_hi=96, sizes=8,
             hq=16, hkv=16, d=128, hidden=2048, dtype="bf16", ratio=0.3, gather="hidden", s_lo=20, s_hi=60),
        # last-token queries over a batch with prompts of more than 128 text tokens
        dict(name="score_last_token", kind="score", batch=64, n_lo=2304, n_hi=3072, t_lo=60, t_hi=142, sizes=9, hq=32,
             hkv=8, d=128, hidden=4096, dtype="bf16", ratio=0.3, gather="hidden", query="last"),
        # keys of one frame
        dict(name="project_frame", kind="project", rows=1536, hidden=2048, out=2048, d=128, bias=False, out8=False),
        # grouped keys of a high-resolution frame with an odd row count, with bias, as 8-bit codes
        dict(name="project_gqa_fp8", kind="project", rows=6157, hidden=3584, out=512, d=128, bias=True, out8=True),
        # keys of a batch
        dict(name="project_batch", kind="project", rows=27648, hidden=4096, out=4096, d=128, bias=False, out8=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step_buffers", "score", "score", "prefill", "full_keys", "project", "project"])
    if kind == "project":
        hidden = rng.choice([256, 896, 1536, 2048, 3584, 4096])
        out = rng.choice([128, 256, 512, 1024, 2048, 3584, 4096])
        rows = min(_log(rng, 40, 40000), _MOST_PROJECT // (hidden * out))
        return dict(kind=kind, rows=rows, hidden=hidden, out=out, d=rng.choice([128, 128, 64, 0]),
                    bias=rng.random() < 0.3, out8=rng.random() < 0.3)
    hq, hkv, d, hidden = rng.choice([(4, 4, 64, 256), (14, 2, 64, 896), (16, 16, 128, 2048), (28, 4, 128, 3584),
                                     (32, 8, 128, 4096), (32, 32, 128, 4096)])
    n_hi = _log(rng, 100, 9000)
    n_lo = n_hi if rng.random() < 0.3 else max(40, int(n_hi * rng.uniform(0.15, 0.95)))
    t_hi = rng.randint(8, 128)
    t_lo = t_hi if n_lo == n_hi and rng.random() < 0.7 else max(1, int(t_hi * rng.uniform(0.3, 1.0)))
    c = dict(kind=kind, batch=_log(rng, 1, 128), n_lo=n_lo, n_hi=n_hi, t_lo=t_lo, t_hi=t_hi, sizes=rng.randrange(1 << 30), hq=hq,
             hkv=hkv, d=d, hidden=hidden, dtype="e4m3" if d == 128 and rng.random() < 0.4 else "bf16",
             ratio=rng.choice([0.1, 0.2, 0.25, 0.3, 0.5, 0.8, 0.9]), gather=rng.choice(["hidden", "hidden+kv"]))
    if kind == "score":
        c["query"] = rng.choice(["all", "all", "last"])
        if c["query"] == "last":
            c["t_hi"] = c["t_hi"] + rng.randint(0, 60)
    if kind in ("full_keys", "prefill"):
        c["s_hi"] = rng.randint(0, 90)
        c["s_lo"] = rng.randint(0, c["s_hi"])
    while c["batch"] > 1 and (work(c)["bytes"] > _MOST_BYTES or c["batch"] * n_hi * t_hi * hq > _MOST_LOGITS):
        c["batch"] -= 1
    return c


def _lens(case):
    """The request lengths of a case: visual, text and system tokens."""
    r = random.Random(case["sizes"])
    n = [r.randint(case["n_lo"], case["n_hi"]) for _ in range(case["batch"])]
    t = [r.randint(case["t_lo"], case["t_hi"]) for _ in range(case["batch"])]
    s = [r.randint(case.get("s_lo", 0), case.get("s_hi", 0)) for _ in range(case["batch"])]
    return n, t, s


def _offsets(lens):
    return np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)


# ----------------------------------------------------------------------------------------------------------- inputs
def _encode(x, dtype, scale=None):
    """bf16 values, or e4m3 codes under one scale (absmax / 448 unless one is given) -> (tensor, scale)."""
    if dtype == "bf16":
        return x.to(torch.bfloat16), 1.0
    if scale is None:
        scale = float(np.float32(float(x.abs().max()) / 448.0))
    return (x / scale).clamp(-448.0, 448.0).to(torch.float8_e4m3fn).view(torch.uint8), scale


def _decode(x, scale):
    return (x if x.dtype == torch.bfloat16 else x.view(torch.float8_e4m3fn)).float().double() * scale


def _scene(case, gen, with_q=True):
    """Queries and keys of a batch. Text queries of a head share a direction (the prompt's topic) beside what each
    token adds; a visual token's keys carry that direction as far as the token matters to the prompt, and token norms
    differ, so the scores spread by an order of magnitude, as attention does."""
    n, t, s = _lens(case)
    hq, hkv, d = case["hq"], case["hkv"], case["d"]
    topic = torch.randn(hkv, d, generator=gen, device="cuda")
    topic /= topic.norm(dim=-1, keepdim=True)

    def rand(*shape):
        return torch.randn(*shape, generator=gen, device="cuda")

    def keys(rows, dtype, scale=None):
        x = rand(rows, hkv, d)
        x *= torch.exp(0.3 * rand(rows, 1, 1))
        x += 3.0 * rand(rows, 1, 1) * topic
        return _encode(x, dtype, scale)

    st = {}
    if with_q:
        q = rand(sum(t), hq, d) + 4.0 * topic.repeat_interleave(hq // hkv, dim=0)
        st["q"], st["q_scale"] = _encode(q, case["dtype"])
        del q
    st["k"], st["k_scale"] = keys(sum(n), case["dtype"])
    if case["kind"] == "full_keys":
        st["k_sys"] = keys(sum(s), case["dtype"], st["k_scale"])[0]
        st["k_txt"] = keys(sum(t), case["dtype"], st["k_scale"])[0]
    return st


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _rows(gen, rows, cols):
    return torch.randn(rows, cols, generator=gen, device="cuda", dtype=torch.float32).to(torch.bfloat16)


def _selector(case, query="all"):
    n, t, _ = _lens(case)
    return select.Selector(case["batch"], sum(n), sum(t), case["hq"], case["hkv"], case["d"], case["dtype"],
                           query=query)


def prepare(case, seed):
    gen = _gen(seed)
    if case["kind"] == "project":
        rows, hidden, out, d = case["rows"], case["hidden"], case["out"], case["d"]
        st = {"case": case, "x": _rows(gen, rows, hidden)}
        gamma = torch.rand(hidden, generator=gen, device="cuda") + 0.5
        w = (torch.randn(out, hidden, generator=gen, device="cuda") / math.sqrt(hidden)).to(torch.bfloat16)
        st["bias"] = torch.randn(out, generator=gen, device="cuda") * 0.1 if case["bias"] else None
        # folded weights and the rotation table are made once per model
        sel = st["sel"] = select.Selector(1, 128, 128, 1, 1, 128, "bf16")
        st["w"] = sel.fold_norm(w, gamma)
        if d:
            st["pos"] = torch.randint(0, 4096, (rows,), generator=gen, device="cuda", dtype=torch.int32)
            st["table"] = sel.rope_table(4096, d, 10000.0)
        else:
            st["pos"] = st["table"] = None
        st["out_scale"] = 5.0 / 448.0 if case["out8"] else 0.0
        return st

    n, t, s = _lens(case)
    st = {"case": case, "so_h": _offsets(n), "to_h": _offsets(t)}
    st["so"], st["to"] = torch.from_numpy(st["so_h"]).cuda(), torch.from_numpy(st["to_h"]).cuda()
    kind = case["kind"]
    st["sel"] = _selector(case, case.get("query", "all"))
    if kind == "prefill":
        # scores as the scoring call leaves them (a mean of probabilities: positive, a long tail)
        st["scores"] = torch.exp(0.8 * torch.randn(sum(n), generator=gen, device="cuda")) / case["n_hi"]
        st["vis"] = _rows(gen, sum(n), case["hidden"])
        st["sys"] = _rows(gen, sum(s), case["hidden"])
        st["txt"] = _rows(gen, sum(t), case["hidden"])
        st["yo_h"] = _offsets(s)
        st["yo"] = torch.from_numpy(st["yo_h"]).cuda()
        return st
    st.update(_scene(case, gen))
    if kind == "full_keys":
        st["yo_h"] = _offsets(s)
        st["yo"] = torch.from_numpy(st["yo_h"]).cuda()
    if kind == "score":
        st["out"] = torch.empty(sum(n), device="cuda")
    if kind in ("step", "step_buffers"):
        st["srcs"] = [_rows(gen, sum(n), case["hidden"])]
        if case["gather"] == "hidden+kv":
            st["srcs"] += [st["k"], _rows(gen, sum(n), case["hkv"] * case["d"]).view(sum(n), case["hkv"], case["d"])]
    if kind == "step_buffers":
        st["keep_h"] = np.array([int(case["ratio"] * x) for x in n], dtype=np.int32)
        st["keep"] = torch.from_numpy(st["keep_h"]).cuda()
        total = st["total"] = int(st["keep_h"].sum())
        st["scores"] = torch.empty(sum(n), device="cuda")
        st["kept"] = torch.empty(max(total, 1), dtype=torch.int32, device="cuda")[:total]
        st["off"] = torch.empty(len(n) + 1, dtype=torch.int32, device="cuda")
        st["off_h"] = np.zeros(len(n) + 1, np.int32)
        st["dsts"] = [torch.empty((total,) + tuple(x.shape[1:]), dtype=x.dtype, device="cuda") for x in st["srcs"]]
        st["row_bytes"] = [x[0].numel() * x.element_size() for x in st["srcs"]]
    return st


# --------------------------------------------------------------------------------------------------------- one pass
def run(st):
    case, sel = st["case"], st["sel"]
    kind = case["kind"]
    if kind == "project":
        return sel.project(st["x"], st["w"], st["bias"], 1e-6, case["d"], st["pos"], st["table"],
                           out_scale=st["out_scale"])
    if kind == "score":
        return sel.score(st["q"], st["to"], st["k"], st["so"], st["q_scale"], st["k_scale"], out=st["out"],
                         text_offsets_h=st["to_h"], seq_offsets_h=st["so_h"])
    if kind == "full_keys":
        scores = sel.score_full_keys(st["q"], st["to"], st["k"], st["so"], st["k_sys"], st["yo"], st["k_txt"],
                                     st["q_scale"], st["k_scale"], text_offsets_h=st["to_h"],
                                     seq_offsets_h=st["so_h"], sys_offsets_h=st["yo_h"])
        kept, off, _ = sel.topk(scores, st["so"], keep_ratio=case["ratio"], seq_offsets_h=st["so_h"])
        return scores, kept, off
    if kind == "prefill":
        kept, off, off_h = sel.topk(st["scores"], st["so"], keep_ratio=case["ratio"], seq_offsets_h=st["so_h"])
        total = int(st["yo_h"][-1] + off_h[-1] + st["to_h"][-1])
        rows = torch.empty(total, case["hidden"], dtype=torch.bfloat16, device="cuda")
        row_off = torch.empty(case["batch"] + 1, dtype=torch.int32, device="cuda")
        pos = torch.empty(total, dtype=torch.int32, device="cuda")
        select.splice(sel.handle, case["batch"], st["sys"], st["yo"], st["yo_h"], st["vis"], st["so"], st["so_h"],
                      kept, off, off_h, st["txt"], st["to"], st["to_h"], 2 * case["hidden"], rows, row_off, pos)
        return kept, rows, row_off, pos
    if kind == "step":
        scores, kept, off, off_h = sel.score_topk(st["q"], st["to"], st["k"], st["so"], st["q_scale"], st["k_scale"],
                                                  keep_ratio=case["ratio"], text_offsets_h=st["to_h"],
                                                  seq_offsets_h=st["so_h"])
        return scores, kept, off, sel.compact(kept, int(off_h[-1]), st["srcs"])
    select.score_topk(sel.handle, case["batch"], st["q"], st["to"], st["to_h"], st["k"], st["so"], st["so_h"],
                      st["q_scale"], st["k_scale"], st["scores"], st["keep"], st["keep_h"], 0.0, st["kept"], st["off"],
                      st["off_h"])
    select.compact(sel.handle, st["total"], st["kept"], int(st["so_h"][-1]), st["srcs"], st["dsts"], st["row_bytes"])
    return st["scores"], st["kept"], st["off"], st["dsts"]


# ------------------------------------------------------------------------------------------- what a pass cannot avoid
def work(case):
    if case["kind"] == "project":
        rows, hidden, out = case["rows"], case["hidden"], case["out"]
        return {"bytes": 2 * rows * hidden + 2 * hidden * out + rows * out * (1 if case["out8"] else 2) +
                (4 * rows if case["d"] else 0), "flops": 2 * rows * hidden * out}
    n, t, s = _lens(case)
    kind, tot = case["kind"], sum(n)
    es = 1 if case["dtype"] == "e4m3" else 2
    kept = sum(int(math.floor(float(np.float32(case["ratio"])) * x)) for x in n)
    row = 2 * case["hidden"]
    if kind == "prefill":
        return {"bytes": 4 * tot + 4 * kept + (2 * row + 4) * (sum(s) + kept + sum(t)), "flops": 0}
    if case.get("query") == "last":
        t = [1] * len(t)
    head = case["d"] * es
    b = tot * case["hkv"] * head + sum(t) * case["hq"] * head + 4 * tot
    f = sum(2 * x * y * case["hq"] * case["d"] for x, y in zip(n, t))
    if kind == "full_keys":
        b += (sum(s) + sum(t)) * case["hkv"] * head
        f += sum(2 * y * (z + (y + 1) // 2) * case["hq"] * case["d"] for y, z in zip(t, s))
    if kind != "score":
        b += 4 * kept
    if kind in ("step", "step_buffers"):
        b += 2 * kept * row
        if case["gather"] == "hidden+kv":
            b += 2 * kept * case["hkv"] * (head + 2 * case["d"])
    return {"bytes": b, "flops": f}


def tolerance(case):
    kind = case["kind"]
    if kind == "prefill":
        return "exact"
    if kind == "project":
        # the result is rounded once to bf16 (2^-9) or to e4m3; sums in another order move a few values by one step
        # (measured against 64 bits: 1.7e-3 and 3.9e-3)
        return {"differ": 1e-3} if case["out8"] else {"rel": 6e-3, "max": 0.016}
    # 32-bit sums of 32-bit exponentials (measured against 64 bits: up to 3.4e-7 and 1.5e-6); two tokens next to each
    # other in rank may change places
    return {"rel": 2e-6, "max": 8e-6, "differ": 0.01}


# ------------------------------------------------------------------------------------------------- the same, in 64 bits
def _exact_scores(st, last=False):
    case = st["case"]
    hq, hkv, d = case["hq"], case["hkv"], case["d"]
    G = hq // hkv
    so, to = st["so_h"], st["to_h"]
    out = torch.empty(int(so[-1]), dtype=torch.float64, device="cuda")
    full = case["kind"] == "full_keys"
    for b in range(case["batch"]):
        t0, t1 = int(to[b + 1]) - 1 if last else int(to[b]), int(to[b + 1])
        T, N = t1 - t0, int(so[b + 1] - so[b])
        q = _decode(st["q"][t0:t1], st["q_scale"]).view(T, hkv, G, d)
        parts = [st["k"][int(so[b]):int(so[b + 1])]]
        S = 0
        if full:
            s0, s1 = int(st["yo_h"][b]), int(st["yo_h"][b + 1])
            S = s1 - s0
            parts += [st["k_sys"][s0:s1], st["k_txt"][t0:t1]]
        k = _decode(torch.cat(parts), st["k_scale"])
        acc = torch.zeros(N, dtype=torch.float64, device="cuda")
        for g in range(hkv):
            x = q[:, g].transpose(0, 1).reshape(G * T, d) @ k[:, g].t() / math.sqrt(d)
            if full:  # text row i sees the text keys 0..i
                later = torch.ones(T, T, dtype=torch.bool, device="cuda").triu(1).repeat(G, 1)
                x[:, N + S:].masked_fill_(later, -math.inf)
            acc += torch.softmax(x, dim=1)[:, :N].sum(dim=0)
        out[int(so[b]):int(so[b + 1])] = acc / (hq * T)
    return out


def exact(case, seed):
    if case["kind"] == "prefill" or case.get("out8"):
        return None
    st = prepare(case, seed)
    if case["kind"] == "project":
        y = torch.empty(case["rows"], case["out"], dtype=torch.float64, device="cuda")
        w, d = st["w"].double(), case["d"]
        for r0 in range(0, case["rows"], 4096):
            x = st["x"][r0:r0 + 4096].double()
            z = torch.rsqrt((x * x).mean(dim=1, keepdim=True) + 1e-6) * (x @ w.t())
            if st["bias"] is not None:
                z += st["bias"].double()
            if d:
                cs = st["table"][st["pos"][r0:r0 + 4096].long()].double()
                c, s = cs[:, None, :, 0], cs[:, None, :, 1]
                z = z.view(-1, case["out"] // d, 2, d // 2)
                z = torch.stack([z[:, :, 0] * c - z[:, :, 1] * s, z[:, :, 1] * c + z[:, :, 0] * s], dim=2)
            y[r0:r0 + 4096] = z.reshape(-1, case["out"])
        return y
    scores = _exact_scores(st, last=case.get("query") == "last")
    if case["kind"] == "score":
        return scores
    if case["kind"] == "full_keys":
        return scores, None, None
    return scores, None, None, [None] * (3 if case["gather"] == "hidden+kv" else 1)
