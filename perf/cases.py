"""The work whose speed is watched, through the package's public entry points.

Three families of calls:

* ``step``: one RPS decoding step (``rps.Step``), from the logits of the base
  prediction and its lookahead branches to the commit decision. Called
  directly, replayed from a CUDA graph as the decode loop replays it, or fed
  from page-locked host memory (``Step.run_host``).
* ``lmhead``: the row statistics straight from hidden states
  (``rps.rps_lmhead_row_stats``), unembedding packed once or row-major.
* ``attention``: the branch-isolating attention of the packed lookahead pass
  (``rps.rps_packed_attention_fwd``).

Sizes are those of the workloads in ``configs`` and of the benchmark; ``draw``
spreads over the ranges between and around them. Inputs come from the seed: the
seeded generator's logits (spikes over noise, three regimes of rows), normal
operands for the two contractions.

A step's ``gain`` and ``margin`` are left out of the outputs: they are
differences of two returned scores, whose relative error says nothing.
"""
import math

import numpy as np
import torch

from paper_2608_11742_gb300 import configs, rps, synth

MIX_A = (0.4, 0.3, 0.3)
MIX_BLOCK = (0.5, 0.3, 0.2)
HEAD_DIM = 128
# No case costs more than the largest listed ones.
MAX_LOGIT_BYTES = 10.6e9
MAX_LM_FLOPS = 2.0 * 1152 * 4096 * 126464
MAX_ATTN_FLOPS = 284e9


def _step(name, n_req, L, V, dtype, P, K, lo, hi, via, k_max=10, low=0.4, mid=0.3):
    """lo..hi: masked positions per request; via: "call", "graph" or "host"; low, mid: shares of the
    one-spike and few-spike rows."""
    c = dict(kind="step", n_req=n_req, L=L, V=V, dtype=dtype, P=P, K=K, lo=lo, hi=hi, via=via, k_max=k_max,
             low=low, mid=mid)
    return dict(name=name, **c) if name else c


def _lm(name, rows, V, d, k, packed):
    c = dict(kind="lmhead", rows=rows, V=V, d=d, k=k, packed=packed)
    return dict(name=name, **c) if name else c


def _attn(name, batch, heads, ctx, branches, length):
    c = dict(kind="attention", batch=batch, heads=heads, ctx=ctx, branches=branches, length=length)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the smallest step: all latency, called directly
        _step("step-tiny", 1, 32, 4096, "f32", 4, 2, 32, 32, "call"),
        # one user decoding a 32-position block, replayed from a graph: the latency of a decode step
        _step("step-one-block", 1, 32, 126464, "bf16", 4, 2, 32, 32, "graph", low=0.5, mid=0.3),
        # one request's generation step, every position masked, called directly
        _step("step-one", 1, 256, 126464, "bf16", 4, 2, 256, 256, "call"),
        # late in the same generation, a tenth masked, the logits in page-locked host memory
        _step("step-host", 1, 256, 126464, "bf16", 4, 2, 26, 26, "host"),
        # fp32 logits, an odd vocabulary with padded rows, ragged masks, longer candidate lists
        _step("step-f32-odd", 3, 96, 32003, "f32", 3, 4, 7, 96, "call", k_max=32),
        # batched serving: ragged masks, NaN in the unmasked rows
        _step("step-serve", 8, 256, 151936, "bf16", 8, 2, 16, 256, "call"),
        # block decoding of many requests, replayed from a graph
        _step("step-blocks", 64, 32, 126464, "bf16", 4, 2, 32, 32, "graph", low=0.5, mid=0.3),
        # LM head and statistics of one block's base rows, row-major unembedding
        _lm("lmhead-block", 32, 126464, 4096, 10, False),
        # ... of a whole generation's base rows
        _lm("lmhead-base", 256, 126464, 4096, 10, True),
        # ... of the lookahead rows (statistics only)
        _lm("lmhead-lookahead", 1152, 126464, 4096, 0, True),
        # lookahead attention of one request's block, ragged against the tiles
        _attn("attention-block", 1, 32, 328, 9, 32),
        # lookahead attention of a batch of generations
        _attn("attention-serve", 8, 32, 512, 9, 256),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "lmhead", "attention"])
    if kind == "step":
        while True:
            V = _log_int(rng, 2000, 152000)
            n_req = _log_int(rng, 1, 64)
            L = rng.choice([32, 48, 64, 128, 256, 384, 512])
            dtype = rng.choice(["bf16", "bf16", "bf16", "f32"])
            P, K = rng.choice([(1, 10), (2, 3), (3, 4), (4, 2), (8, 2)])
            if n_req * (1 + P * K) * L * V * (2 if dtype == "bf16" else 4) <= MAX_LOGIT_BYTES:
                break
        hi = rng.choice([L, L, max(2, L // 2), max(2, L // 10)])
        lo = rng.choice([hi, max(1, hi // 16)])
        low = rng.choice([0.3, 0.4, 0.5])
        return _step(None, n_req, L, V, dtype, P, K, lo, hi, rng.choice(["call", "graph"]),
                     rng.choice([10, 10, 16, 32]), low, 0.3)
    if kind == "lmhead":
        while True:
            rows, V = _log_int(rng, 4, 1408), _log_int(rng, 8000, 152000)
            d = 64 * rng.randint(16, 64)
            if 2.0 * rows * V * d <= MAX_LM_FLOPS:
                break
        return _lm(None, rows, V, d, rng.choice([0, 10, 10, 20]), rng.choice([True, False]))
    while True:
        c = _attn(None, rng.randint(1, 8), rng.choice([8, 16, 28, 32]), 8 * rng.randint(0, 256), rng.randint(2, 17),
                  8 * _log_int(rng, 3, 64))
        if work(c)["flops"] <= MAX_ATTN_FLOPS:
            return c


# ---------------------------------------------------------------- step
def _params(case):
    ex = configs.EXERCISE
    return configs.Params(case["k_max"], ex.r, ex.tau_pivot, ex.tau, ex.lam, case["P"], case["K"])


def _mixture(case):
    return (case["low"], case["mid"], 1.0 - case["low"] - case["mid"])


def _masks(case, seed):
    n, L = case["n_req"], case["L"]
    pos = np.full((n, L), -1, dtype=np.int32)
    cnt = np.zeros(n, dtype=np.int32)
    valid = np.zeros((n, L), dtype=np.uint8)
    for q in range(n):
        c = synth.ragged_count(seed, q, case["lo"], case["hi"])
        p = synth.masked_positions(seed, q, L, c)
        pos[q, :c], cnt[q], valid[q, p] = p, c, 1
    return pos, cnt, valid


def _logits(case, seed):
    """[n_req][1 + P K][L][V] on the GPU, rows padded to 16 bytes, unmasked rows NaN; and the mask."""
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    unit = 16 // dt.itemsize
    pitch = -(-case["V"] // unit) * unit
    full = torch.empty((case["n_req"], 1 + case["P"] * case["K"], case["L"], pitch), dtype=dt, device="cuda")
    pos, cnt, valid = _masks(case, seed)
    z = full[..., : case["V"]]
    synth.device_fill(z, seed, _mixture(case), valid=torch.from_numpy(valid).cuda())
    return z, torch.from_numpy(pos).cuda(), torch.from_numpy(cnt).cuda()


def _prepare_step(case, seed):
    z, pos, cnt = _logits(case, seed)
    s = {"case": case, "pos": pos, "cnt": cnt, "z": z,
         "step": rps.Step(case["n_req"], case["L"], case["V"], _params(case), "cuda", z.dtype)}
    if case["via"] == "host":
        s["host"] = torch.empty(z.shape, dtype=z.dtype, pin_memory=True)
        s["host"].copy_(z)
        s["z"] = torch.zeros_like(z)
    elif case["via"] == "graph":
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            s["step"].run(z, pos, cnt)
        torch.cuda.current_stream().wait_stream(side)
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            s["step"].run(z, pos, cnt)
    return s


_STATS = ("zmax", "lse", "H", "pmax", "argmax")
_TOPK = ("mu", "htrunc", "topk_idx", "topk_logit")
_PIVOTS = ("state", "n_commit", "commit_pos", "commit_tok", "pivot_pos", "n_cand", "cand_tok", "n_branch_rows",
           "branch_rows")
_SCORES = ("mean_H", "n_tau", "log_a", "score")
_COMMIT = ("best_slot", "winner", "commit_pos", "commit_tok", "mask_pos", "mask_cnt")


def _run_step(s):
    st = s["step"]
    if s["case"]["via"] == "host":
        st.run_host(s["host"], s["z"], s["pos"], s["cnt"])
    elif s["case"]["via"] == "graph":
        s["graph"].replay()
    else:
        st.run(s["z"], s["pos"], s["cnt"])
    return {"base": {f: getattr(st.base, f) for f in _STATS + _TOPK},
            "branch": {f: getattr(st.branch, f) for f in _STATS},
            "pivots": {f: getattr(st.piv, f) for f in _PIVOTS},
            "scores": {f: getattr(st.scores, f) for f in _SCORES},
            "commit": {f: getattr(st.commit, f) for f in _COMMIT}}


def _row_stats64(z):
    """zmax, lse, H, pmax of rows z (exact in fp64), and log p."""
    x = z.double()
    lse = torch.logsumexp(x, 1)
    logp = x - lse[:, None]
    return x.amax(1), lse, -(logp.exp() * logp).sum(1), logp.amax(1).exp()


def _rows_stats64(z, rows):
    out = []
    per = max(1, int(2e8) // z.shape[-1])
    for i in range(0, len(rows), per):
        r = torch.as_tensor(rows[i:i + per], device="cuda", dtype=torch.long).reshape(-1, 3)
        out.append(torch.stack(_row_stats64(z[r[:, 0], r[:, 1], r[:, 2]]), 1).cpu().numpy())
    return np.concatenate(out) if out else np.zeros((0, 4))


def _topk_rows(z, k):
    """The k largest logits of fp32 rows in rank order (logit descending, then token ascending)."""
    b = z.contiguous().view(torch.int32)
    key = torch.where(b < 0, b ^ 0x7FFFFFFF, b).long() * (1 << 32) - torch.arange(z.shape[1], device=z.device)
    idx = torch.topk(key, k, dim=1).indices
    return idx, torch.gather(z, 1, idx)


def _exact_step(case, seed):
    z, pos_t, cnt_t = _logits(case, seed)
    pos, cnt, prm = pos_t.cpu().numpy(), cnt_t.cpu().numpy(), _params(case)
    n, L, P, K, k = case["n_req"], case["L"], case["P"], case["K"], case["k_max"]
    NB = P * K
    nan = lambda *s: np.full(s, np.nan)  # noqa: E731
    base = {f: nan(n * L) for f in ("zmax", "lse", "H", "pmax", "mu", "htrunc")}
    base["topk_logit"] = nan(n * L, k)
    branch = {f: nan(n * NB * L) for f in ("zmax", "lse", "H", "pmax")}
    scores = {f: nan(n, P, K + 1) for f in ("mean_H", "log_a", "score")}
    rows, slots = [], []
    for q in range(n):
        rows += [(q, 0, int(p)) for p in pos[q, : cnt[q]]]
        slots += list(range(q * L, q * L + int(cnt[q])))
    st = _rows_stats64(z, rows)
    slots = np.array(slots, dtype=np.int64)
    for i, f in enumerate(("zmax", "lse", "H", "pmax")):
        base[f][slots] = st[:, i]
    per = max(1, int(1e8) // case["V"])
    topk_idx = np.zeros((n * L, k), dtype=np.int64)
    for i in range(0, len(rows), per):
        r = torch.as_tensor(rows[i:i + per], device="cuda")
        idx, val = _topk_rows(z[r[:, 0], r[:, 1], r[:, 2]].float(), k)
        lp = val.double() - torch.as_tensor(st[i:i + per, 1], device="cuda")[:, None]
        base["mu"][slots[i:i + per]] = lp.exp().sum(1).cpu().numpy()
        base["htrunc"][slots[i:i + per]] = -(lp.exp() * lp).sum(1).cpu().numpy()
        base["topk_logit"][slots[i:i + per]] = val.double().cpu().numpy()
        topk_idx[slots[i:i + per]] = idx.cpu().numpy()
    # standard commit, pivots, candidates, lookahead rows
    tau, log_r = float(np.float32(prm.tau)), math.log(float(np.float32(prm.r)))
    look, look_slots, todo = [], [], []
    for q in range(n):
        b = slice(q * L, q * L + int(cnt[q]))
        pm, ht, mu = base["pmax"][b], base["htrunc"][b], base["mu"][b]
        commit = pm >= tau
        if cnt[q] and not commit.any():
            commit[np.lexsort((pos[q, : cnt[q]], -pm))[0]] = True
        rem = np.flatnonzero(~commit)
        feasible = rem[mu[rem] >= prm.tau_pivot]
        piv = feasible[np.lexsort((pos[q, feasible], -ht[feasible]))][:P]
        off = 0
        for j, i in enumerate(piv):
            tl = base["topk_logit"][q * L + i]
            cand = np.flatnonzero(tl - base["zmax"][q * L + i] >= log_r)[:K]
            if len(cand) < 2:
                continue
            d_j = rem[rem != i]
            todo.append((q, j, K, q * L + i, tl[0], None, d_j))
            for c in range(len(cand)):
                first = q * NB * L + off
                look += [(q, 1 + j * K + c, int(pos[q, x])) for x in d_j]
                look_slots += list(range(first, first + len(d_j)))
                todo.append((q, j, c, q * L + i, tl[cand[c]], first, d_j))
                off += len(d_j)
    st = _rows_stats64(z, look)
    look_slots = np.array(look_slots, dtype=np.int64)
    for i, f in enumerate(("zmax", "lse", "H", "pmax")):
        branch[f][look_slots] = st[:, i]
    for q, j, c, row, zc, first, d_j in todo:
        h = base["H"][q * L + d_j] if first is None else branch["H"][first:first + len(d_j)]
        mean = float(h.mean()) if len(h) else 0.0
        la = zc - base["lse"][row]
        scores["mean_H"][q, j, c], scores["log_a"][q, j, c] = mean, la
        scores["score"][q, j, c] = -mean + float(np.float32(prm.lam)) * la
    return {"base": {f: base.get(f) for f in _STATS + _TOPK}, "branch": {f: branch.get(f) for f in _STATS},
            "pivots": {f: None for f in _PIVOTS}, "scores": {f: scores.get(f) for f in _SCORES},
            "commit": {f: None for f in _COMMIT}}


def _work_step(case):
    """Rows scored in expectation: the masked base rows, then P K branches of the rows that stay masked."""
    m = (case["lo"] + case["hi"]) / 2.0
    left = max(0.0, m * (1.0 - case["low"]) - 1.0)
    rows = case["n_req"] * (m + case["P"] * case["K"] * left)
    return {"bytes": rows * (case["V"] * (2 if case["dtype"] == "bf16" else 4) + 20) + 8.0 * m * case["n_req"] * case["k_max"],
            "flops": 0}


# ---------------------------------------------------------------- LM head
def _lm_inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    h = torch.randn((case["rows"], case["d"]), generator=g, device="cuda").bfloat16()
    w = torch.empty((case["V"], case["d"]), dtype=torch.bfloat16, device="cuda").normal_(
        0.0, 3.0 / math.sqrt(case["d"]), generator=g)  # logits of about 3 nats' spread, as a model's
    return h, w


def _prepare_lm(case, seed):
    h, w = _lm_inputs(case, seed)
    ws = torch.empty(rps.rps_lmhead_workspace_bytes(case["rows"], case["V"], case["k"]), dtype=torch.uint8,
                     device="cuda")
    rps.rps_workspace_init(ws)
    return {"case": case, "h": h, "w": w, "ws": ws, "prm": configs.Params(k_max=max(1, case["k"])),
            "packed": rps.rps_lmhead_pack_unembed(w) if case["packed"] else None,
            "out": rps.RowStatsBuf.alloc(case["rows"], case["k"], "cuda")}


def _run_lm(s):
    rps.rps_lmhead_row_stats(s["h"], s["w"], s["prm"], s["out"], s["ws"], packed=s["packed"])
    return {f: getattr(s["out"], f) for f in (_STATS + _TOPK if s["case"]["k"] else _STATS)}


def _exact_lm(case, seed):
    h, w = _lm_inputs(case, seed)
    z = torch.empty((case["rows"], case["V"]), dtype=torch.float64, device="cuda")
    for v in range(0, case["V"], 16384):
        z[:, v:v + 16384] = h.double() @ w[v:v + 16384].double().T
    zmax, lse, H, pmax = _row_stats64(z)
    out = dict(zmax=zmax, lse=lse, H=H, pmax=pmax, argmax=None)
    if case["k"]:
        val = torch.topk(z, case["k"], dim=1).values
        lp = val - lse[:, None]
        out.update(mu=lp.exp().sum(1), htrunc=-(lp.exp() * lp).sum(1), topk_idx=None, topk_logit=val)
    return out


def _work_lm(case):
    return {"bytes": 2.0 * case["V"] * case["d"] + 2.0 * case["rows"] * case["d"] + case["rows"] * (20 + 8 * case["k"]),
            "flops": 2.0 * case["rows"] * case["V"] * case["d"]}


# ---------------------------------------------------------------- attention
def _attn_inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    n = case["ctx"] + case["branches"] * case["length"]
    shape = (case["batch"], case["heads"], n, HEAD_DIM)
    q = (2.0 * torch.randn(shape, generator=g, device="cuda")).bfloat16()  # scores of about 2 nats' spread
    k = torch.randn(shape, generator=g, device="cuda").bfloat16()
    v = torch.randn(shape, generator=g, device="cuda").bfloat16()
    return q, k, v


def _prepare_attn(case, seed):
    q, k, v = _attn_inputs(case, seed)
    return {"case": case, "q": q, "k": k, "vt": v.transpose(2, 3).contiguous(), "out": torch.zeros_like(q)}


def _run_attn(s):
    c = s["case"]
    rps.rps_packed_attention_fwd(s["q"], s["k"], s["vt"], s["out"], c["ctx"], c["branches"], c["length"],
                                 HEAD_DIM ** -0.5)
    return s["out"]


def _exact_attn(case, seed):
    q, k, v = _attn_inputs(case, seed)
    scale = float(np.float32(HEAD_DIM ** -0.5))
    out = torch.empty(q.shape, dtype=torch.float64, device="cuda")
    c, length = case["ctx"], case["length"]
    for b in range(case["batch"]):
        qb, kb, vb = q[b].double(), k[b].double(), v[b].double()

        def attend(rows, branch):
            own = slice(c + branch * length, c + (branch + 1) * length)
            keys, vals = torch.cat((kb[:, :c], kb[:, own]), 1), torch.cat((vb[:, :c], vb[:, own]), 1)
            out[b, :, rows] = torch.softmax(scale * (qb[:, rows] @ keys.transpose(1, 2)), 2) @ vals

        if c:
            attend(slice(0, c), 0)
        for j in range(case["branches"]):
            attend(slice(c + j * length, c + (j + 1) * length), j)
    return out


def _work_attn(case):
    n, seen = case["ctx"] + case["branches"] * case["length"], case["ctx"] + case["length"]
    return {"bytes": 4.0 * case["batch"] * case["heads"] * n * HEAD_DIM * 2,
            "flops": 4.0 * HEAD_DIM * case["batch"] * case["heads"] * n * seen}


# ---------------------------------------------------------------- the cases' functions
def prepare(case, seed):
    return {"step": _prepare_step, "lmhead": _prepare_lm, "attention": _prepare_attn}[case["kind"]](case, seed)


def run(state):
    return {"step": _run_step, "lmhead": _run_lm, "attention": _run_attn}[state["case"]["kind"]](state)


def exact(case, seed):
    return {"step": _exact_step, "lmhead": _exact_lm, "attention": _exact_attn}[case["kind"]](case, seed)


def work(case):
    return {"step": _work_step, "lmhead": _work_lm, "attention": _work_attn}[case["kind"]](case)


def tolerance(case):
    # about four times the error of each path against exact(), largest over its outputs
    if case["kind"] == "step":  # fp32 sums over a row (5e-7); decisions and ranks are exact
        return {"rel": 2e-6, "max": 2e-5, "differ": 0.0}
    if case["kind"] == "lmhead":  # fp32 accumulation over d (2e-5 in p); near-equal logits may swap ranks
        return {"rel": 8e-5, "max": 1e-3, "differ": 0.005}
    return {"rel": 1e-2, "max": 0.1}  # bf16 probabilities and output (2e-3)
