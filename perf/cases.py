"""Performance cases of the restore-and-resume library, all through its public entry points.

A case is one call as an engine makes it on its stream: the linear-attention prefill of the
tails or decode steps of a batch of requests (padded, packed, or segment-parallel), the
restore of one resumed request, or one tensor-parallel rank's transfer of its KV heads.  A
(request, linear layer) pair is one problem of a prefill call, so a call covers every linear
layer of its requests, as the library is meant to be used.

Sizes follow the repository's workloads: the tiny stack (2 heads, d = 64, log-sigmoid gates),
the hybrid stack (9 linear layers of 16 heads, d = 128, checkpoints every 256 tokens; 3 full
layers of 4 KV heads, pages of 16 tokens), the single-layer sweep (16 heads, checkpoints every
512) and the long-context layer (4 requests of 32 heads).
"""
import math
import random

import torch

import paper_2609_15030_gb300 as hs

DEV = "cuda:0"


# ---- the cases ---------------------------------------------------------------------------


def _linear(name, op, requests, layers, heads, d, tokens, start, interval, gates):
    """A linear-attention call.  tokens / start: (lowest, highest) per request; start points
    are multiples of `grid` (a resume point is a checkpoint position)."""
    return {"name": name, "op": op, "requests": requests, "layers": layers, "heads": heads, "d": d,
            "tokens_lo": tokens[0], "tokens_hi": tokens[1], "start_lo": start[0],
            "start_hi": start[1], "grid": start[2], "interval": interval, "gates": gates,
            "lens": 1}


def listed():
    return [
        # the smallest prefill: one layer of the tiny stack resumed at 192 of 256 tokens
        _linear("tiny_tail", "prefill", 1, 1, 2, 64, (64, 64), (192, 192, 64), 64, "sigmoid"),
        # one decode step of one request, all linear layers of the hybrid stack
        _linear("decode_one", "prefill", 1, 9, 16, 128, (1, 1), (4608, 4700, 1), 256, "uniform"),
        # one decode step of a serving batch: 32 requests at different positions
        _linear("decode_batch", "prefill", 32, 9, 16, 128, (1, 1), (1, 8000, 1), 256, "uniform"),
        # short suffixes after a full cache hit (or draft tokens to verify), ragged
        _linear("short_suffixes", "prefill", 8, 9, 16, 128, (2, 8), (200, 5000, 1), 256,
                "uniform"),
        # the resumed 256-token tail of one hybrid-stack request of 4,608 tokens
        _linear("tail_hybrid", "prefill", 1, 9, 16, 128, (256, 256), (4352, 4352, 256), 256,
                "uniform"),
        # an odd-length tail whose gates decay fast (log-sigmoid gates, as in the tiny stack)
        _linear("tail_decaying", "prefill", 1, 9, 16, 128, (475, 475), (4096, 4096, 256), 256,
                "sigmoid"),
        # one engine batch of nine requests' tails, unpadded
        _linear("tails_packed", "packed", 9, 9, 16, 128, (65, 512), (0, 4096, 256), 256,
                "uniform"),
        # the largest: recomputation of four 16k-token prompts, one long-context layer
        _linear("recompute_long", "prefill", 4, 1, 32, 128, (16384, 16384), (0, 0, 512), 512,
                "uniform"),
        # few problems, segment-parallel: a resumed 512-token tail on the fixed workspace ...
        _linear("scan_tail", "noalloc", 1, 1, 16, 128, (512, 512), (4096, 4096, 512), 512,
                "uniform"),
        # ... and the recomputation of a 4,608-token prompt on the caller's workspace
        _linear("scan_recompute", "scan", 1, 1, 16, 128, (4608, 4608), (0, 0, 512), 512,
                "uniform"),
        # KV pages and states of one resumed request of the hybrid stack (4,352 cached tokens)
        {"name": "restore_request", "op": "restore", "layers": 3, "pages": 272,
         "page_bytes": 32768, "blocks": 4096, "slots": 9, "floats": 262144},
        # one of four tensor-parallel ranks saves its 2 of 8 FP8 KV heads of 4,096 tokens
        {"name": "save_rank_slice", "op": "slices", "save": True, "layers": 48, "pages": 256,
         "rows": 32, "row_bytes": 1024, "off": 256, "cols": 256, "blocks": 1024},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["prefill", "prefill", "decode", "short", "packed", "scan", "noalloc",
                     "restore", "slices"])
    if op == "restore":
        pages = _log_int(rng, 4, 2032)
        return {"op": "restore", "layers": rng.randint(1, 12), "pages": pages,
                "page_bytes": 1024 * rng.choice([8, 16, 32, 64]), "blocks": pages + rng.randint(0, 2048),
                "slots": rng.randint(1, 36), "floats": 128 * 128 * rng.choice([2, 8, 16, 32])}
    if op == "slices":
        heads, ranks, width = rng.choice([4, 8]), rng.choice([2, 4]), rng.choice([64, 128, 256])
        cols = heads // ranks * width
        pages = _log_int(rng, 4, 1024)
        return {"op": "slices", "save": rng.random() < 0.5, "layers": rng.randint(1, 48),
                "pages": pages, "rows": 2 * rng.choice([16, 32]), "row_bytes": heads * width,
                "off": cols * rng.randint(0, ranks - 1), "cols": cols,
                "blocks": pages + rng.randint(0, 512)}
    d = rng.choice([64, 128, 128, 128])
    heads = rng.choice([2, 4, 8, 16, 16, 32])
    interval = rng.choice([0, 64, 128, 256, 512])
    gates = rng.choice(["uniform", "uniform", "sigmoid"])
    grid = interval if interval and rng.random() < 0.7 else 1
    start = (0, _log_int(rng, 64, 32768), grid)
    if op == "decode":
        layers = rng.randint(1, 18)
        tokens, requests = (1, 1), _log_int(rng, 1, min(64, 384 // layers))
        start, op = (1, 32768, 1), "prefill"
    elif op == "short":
        layers = rng.randint(1, 18)
        tokens, requests = (1, rng.randint(2, 8)), _log_int(rng, 1, min(16, 384 // layers))
        start, op = (1, 32768, 1), "prefill"
    elif op in ("prefill", "packed"):
        layers = rng.randint(1, 18)
        requests = _log_int(rng, 1, 12)
        most = max(9, min(8192, 1_500_000 // (requests * layers * heads)))
        hi = _log_int(rng, 9, most)
        tokens = (hi, hi) if op == "prefill" and rng.random() < 0.5 else (max(9, hi // 8), hi)
    else:
        layers, requests, heads = 1, rng.choice([1, 1, 2]), min(heads, 16)
        hi = _log_int(rng, 33, 8192)
        if op == "noalloc":     # the segments' two states fit the fixed workspace
            fit = hs.HS_NOALLOC_SCRATCH_BYTES // (2 * requests * heads * d * d * 4)
            hi = max(33, min(hi, 64 * (fit - 1)))
        tokens = (hi, hi)
    case = _linear("", op, requests, layers, heads, d, tokens, start, interval, gates)
    del case["name"]
    case["lens"] = rng.randint(1, 1 << 20)
    return case


# ---- sizes -------------------------------------------------------------------------------


def _positions(case):
    """pos0 and n_tokens of every problem: a request's layers share them."""
    r = random.Random(case["lens"])
    pos0, n = [], []
    for _ in range(case["requests"]):
        g = case["grid"]
        p = g * r.randint(-(-case["start_lo"] // g), max(-(-case["start_lo"] // g), case["start_hi"] // g))
        t = r.randint(case["tokens_lo"], case["tokens_hi"])
        pos0 += [p] * case["layers"]
        n += [t] * case["layers"]
    return pos0, n


def _checkpoints(case):
    """(problem, tokens done) of every checkpoint, in the order of the slots."""
    c = case["interval"]
    return [(b, m * c - p) for b, (p, n) in enumerate(zip(*_positions(case))) if c
            for m in range(p // c + 1, (p + n) // c + 1)]


def _rows(case, n):
    """First row of every problem and the number of rows of q, k, v, the gates and o."""
    if case["op"] == "packed":
        cu = [0]
        for x in n:
            cu.append(cu[-1] + x)
        return cu[:-1], cu[-1]
    T = max(n)
    return [b * T for b in range(len(n))], len(n) * T


def work(case):
    if case["op"] == "restore":
        return {"bytes": 2 * (case["layers"] * case["pages"] * case["page_bytes"]
                              + case["slots"] * case["floats"] * 4), "flops": 0}
    if case["op"] == "slices":
        return {"bytes": 2 * case["layers"] * case["pages"] * case["rows"] * case["cols"], "flops": 0}
    _, n = _positions(case)
    h, d = case["heads"], case["d"]
    # q, k, v in bf16, the gates and o in float32; the state in and out; the checkpoints
    return {"bytes": sum(n) * h * d * 14 + (2 * len(n) + len(_checkpoints(case))) * h * d * d * 4,
            "flops": sum(n) * h * 5 * d * d}


# ---- one pass ----------------------------------------------------------------------------


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def prepare(case, seed):
    g = _gen(seed)
    if case["op"] == "restore":
        L, P, pb, nb = case["layers"], case["pages"], case["page_bytes"], case["blocks"]
        s = {"case": case,
             "staging": torch.randint(0, 256, (L, P, pb), dtype=torch.uint8, device=DEV, generator=g),
             "cache": torch.zeros((L, nb, pb), dtype=torch.uint8, device=DEV),
             "table": torch.randperm(nb, device=DEV, generator=g)[:P].int(),
             "slots": torch.randn((case["slots"], case["floats"]), device=DEV, generator=g),
             "live": torch.zeros((case["slots"], case["floats"]), device=DEV)}
        for name in ("staging", "cache", "slots", "live"):
            s[name + "_ptrs"] = hs.ptr_array(list(s[name]), DEV)
        return s
    if case["op"] == "slices":
        L, P, nb = case["layers"], case["pages"], case["blocks"]
        page = case["rows"] * case["row_bytes"]
        full, part = (L, nb, page), (L, P, case["rows"] * case["cols"])

        def data(shape, random_bytes):
            if random_bytes:
                return torch.randint(0, 256, shape, dtype=torch.uint8, device=DEV, generator=g)
            return torch.zeros(shape, dtype=torch.uint8, device=DEV)
        s = {"case": case, "cache": data(full, case["save"]), "staging": data(part, not case["save"]),
             "table": torch.randperm(nb, device=DEV, generator=g)[:P].int()}
        for name in ("staging", "cache"):
            s[name + "_ptrs"] = hs.ptr_array(list(s[name]), DEV)
        return s
    pos0, n = _positions(case)
    h, d = case["heads"], case["d"]
    first, rows = _rows(case, n)
    shape = (rows, h, d)

    def normal():
        return torch.randn(shape, device=DEV, generator=g)
    if case["gates"] == "sigmoid":      # q, k, v ~ N(0,1)/8, gates log sigmoid(N(2, 0.5))
        q, k, v = ((normal() / 8).bfloat16() for _ in range(3))
        a = torch.nn.functional.logsigmoid(normal() * 0.5 + 2.0)
    else:                               # k normalised per token and head, gates U(-0.1, 0)
        q, k, v = normal() / math.sqrt(d), normal(), normal() / math.sqrt(d)
        q, k, v = q.bfloat16(), (k / k.norm(dim=-1, keepdim=True)).bfloat16(), v.bfloat16()
        a = torch.rand(shape, device=DEV, generator=g) * -0.1
    # a recomputation starts from the zero state, a resumed tail from a restored one
    scale = 0.0 if case["start_hi"] == 0 else 0.1
    state = torch.randn((len(n), h, d, d), device=DEV, generator=g) * scale
    ck = len(_checkpoints(case))
    s = {"case": case, "q": q, "k": k, "v": v, "a": a, "o": torch.zeros(shape, device=DEV),
         "state": state, "pos0": pos0, "n": n, "ckpt": torch.zeros((ck, h, d, d), device=DEV)}
    s["ckpt_ptrs"] = hs.ptr_array(list(s["ckpt"]), DEV) if ck else None
    s["shape"] = hs.make_shape(len(n), h, d, d, max(n))
    if case["op"] == "packed":
        s["cu"] = first + [rows]
    if case["op"] == "scan":
        s["ws_bytes"] = hs.hs_linattn_scan_workspace_bytes(s["shape"], pos0, n)
        s["ws"] = torch.empty(s["ws_bytes"] // 4, device=DEV)
    return s


def run(s):
    case = s["case"]
    op = case["op"]
    if op == "restore":
        hs.hs_restore_request(s["staging_ptrs"], s["cache_ptrs"], case["layers"], s["table"],
                              case["pages"], case["page_bytes"], case["blocks"], s["slots_ptrs"],
                              s["live_ptrs"], case["slots"], case["floats"])
        return {"cache": s["cache"], "live": s["live"]}
    if op == "slices":
        call, src, dst = ((hs.hs_save_kv_page_slices, "cache", "staging") if case["save"] else
                          (hs.hs_restore_kv_page_slices, "staging", "cache"))
        call(s[src + "_ptrs"], s[dst + "_ptrs"], case["layers"], s["table"], case["pages"],
             case["rows"] * case["row_bytes"], case["rows"], case["off"], case["cols"], case["blocks"])
        return {dst: s[dst]}
    args = (s["shape"], s["q"], s["k"], s["v"], s["a"], s["o"], s["state"], s["pos0"], s["n"])
    interval = case["interval"]
    if op == "prefill":
        hs.hs_linattn_prefill_from_state(*args, interval, s["ckpt_ptrs"])
    elif op == "packed":
        hs.hs_linattn_prefill_packed(*args, s["cu"], interval, s["ckpt_ptrs"])
    elif op == "scan":
        hs.hs_linattn_prefill_scan(*args, interval, s["ckpt_ptrs"], s["ws"], s["ws_bytes"])
    else:
        hs.hs_linattn_prefill_scan_noalloc(*args, interval, s["ckpt_ptrs"])
    out = {"o": s["o"], "state": s["state"]}
    if s["ckpt"].numel():
        out["ckpt"] = s["ckpt"]
    return out


# ---- what is right -----------------------------------------------------------------------


def tolerance(case):
    if case["op"] in ("restore", "slices"):
        return "exact"
    if case["tokens_hi"] <= 8 and case["op"] in ("prefill", "packed"):
        return {"rel": 1e-6, "max": 2e-5}    # float32 token by token: 1.2e-7 from float64 measured
    # 11-bit tensor-core operands, float32 sums: 2e-4 to 3.5e-4 from float64 measured
    return {"rel": 1.5e-3, "max": 2e-2}


def exact(case, seed):
    """The recurrence token by token in float64: S <- diag(exp(a)) S + k v^T, o = q S."""
    if case["op"] in ("restore", "slices"):
        return None
    if case["tokens_hi"] * case["requests"] * case["layers"] * case["heads"] > 40_000_000:
        return None
    s = prepare(case, seed)
    n = s["n"]
    first, _ = _rows(case, n)
    f8 = torch.float64
    S = s["state"].to(f8)
    o = torch.zeros(s["o"].shape, dtype=f8, device=DEV)
    ckpt = torch.zeros(s["ckpt"].shape, dtype=f8, device=DEV)
    due = {}
    for i, (b, t) in enumerate(_checkpoints(case)):
        due.setdefault(t, []).append((i, b))
    first_t, n_t = torch.tensor(first, device=DEV), torch.tensor(n, device=DEV)
    steady = min(n)
    for t in range(max(n)):
        rows = first_t + t
        if t < steady:
            live = slice(None)
        else:                       # the problems that still have a token
            live = (n_t > t).nonzero().squeeze(1)
            rows = rows[live]
        q, k, v, a = (s[x][rows].to(f8) for x in ("q", "k", "v", "a"))
        St = S[live] * a.exp().unsqueeze(-1)
        St += k.unsqueeze(-1) * v.unsqueeze(-2)
        S[live] = St
        o[rows] = torch.matmul(q.unsqueeze(-2), St).squeeze(-2)
        for i, b in due.get(t + 1, ()):
            ckpt[i] = S[b]
    out = {"o": o, "state": S}
    if ckpt.numel():
        out["ckpt"] = ckpt
    return out
