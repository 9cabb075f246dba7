"""The work that users of this library have it do, as timed cases.

A case is a dict of plain sizes and options.  `prepare` builds what a program holds before the call (paged pool,
block tables, queries, a `Compressor` or `HostStepRunner` with its buffers), `run` makes one pass through the public
entry points.  Four kinds:

  step     the compression step, one `actkv_step_device` call (HostStepRunner.run_device) or, with host = True, one
           `actkv_step_host` call from pinned host buffers: [monitor ->] LSE -> pooled score -> TopK -> fresh pages
  stream   the per-decode-step score update (`actkv_score_accumulate`), one action query per request
  monitor  the confidence monitor and budget update (`actkv_budget`) on the logits of newly decoded tokens
  region   the end of an action region in the streaming mode: LRFU keep-score update and TopK on the running score,
           in-place tail compaction, keep-scores of the survivors (Compressor methods of the same names)

A compression step rewrites the block tables.  A serving program uploads its tables before each step; `run` copies
them from a packed device buffer for the same effect, so that every pass starts from the same cache.
"""
import math
import random

import torch

from paper_2609_31395_b200 import binding as B
from paper_2609_31395_b200 import harness as H
from paper_2609_31395_b200 import synth

DEV = "cuda:0"
VOCAB = 151936

STEP = dict(kind="step", layers=1, kv_heads=8, group=4, head_dim=128, page=16, requests=1, len_lo=4096, len_hi=4096,
            win_lo=32, win_hi=32, keep=0.25, causal=False, lse="computed", layers_per_call=0, logit_rows=0,
            clamp_lo=0.0, clamp_hi=0.0, tables="permutation", topics=0, host=False, shape=1)
STREAM = dict(kind="stream", layers=1, kv_heads=8, group=4, head_dim=128, page=16, requests=8, len_lo=8192,
              len_hi=8192, shape=1)
MONITOR = dict(kind="monitor", requests=16, rows_lo=1, rows_hi=1, history=512, vocab=VOCAB, shape=1)
REGION = dict(kind="region", layers=8, kv_heads=8, group=4, head_dim=128, page=16, requests=16, len_lo=8192,
              len_hi=24576, keep=0.8, protect=1024, shape=1)


def listed():
    return [
        # The smallest whole step: one layer of 8 KV heads, one 4096-token request cut to 1024 (the single-layer
        # configuration, and the kernel-table shapes with one request).  A call per layer inside an attention hook
        # looks like this; latency and launches count.
        dict(STEP, name="step_4k_x1"),
        # The kernel-table shape 2048 -> 1536 with 16 requests: one layer, the attention backend hands over the LSE.
        dict(STEP, name="step_2k_x16_lse", requests=16, len_lo=2048, len_hi=2048, keep=0.75, lse="supplied",
             tables="fragmented"),
        # One long request on all 36 layers of the 8B attention shape (32768 tokens, window 64, 25 % kept).
        dict(STEP, name="step_32k_x1", layers=36, len_lo=32768, len_hi=32768, win_lo=64, win_hi=64, tables="fragmented"),
        # The benchmark workload: 48 layers, 8 requests x 35000 tokens, window 64, 26 % kept, budgets from 64 logit
        # rows per request, copies of a layer group inside the next one's score kernel.  The largest call.
        dict(STEP, name="step_35k_x8", layers=48, kv_heads=4, group=8, requests=8, len_lo=35000, len_hi=35000, win_lo=64,
             win_hi=64, keep=0.26, layers_per_call=16, logit_rows=64, clamp_lo=0.26, clamp_hi=0.26, tables="interleaved",
             topics=64),
        # The serving mix: 64 requests of 8K-64K tokens in a shared fragmented pool, budgets from the monitor within
        # 15-40 %, LSE from the attention backend; four layers, one group of a pipelined server.
        dict(STEP, name="serving_mix_x64", layers=4, kv_heads=4, group=8, requests=64, len_lo=8192, len_hi=65536,
             win_lo=64, win_hi=64, keep=0.2, lse="supplied", logit_rows=32, clamp_lo=0.15, clamp_hi=0.40,
             tables="fragmented", topics=64, shape=4),
        # One round of the iterative agent trace: 16 requests, causal windows of 32-96 action tokens at the end of a
        # 12K-20K cache of which most is kept, so that copies weigh as much as scores.
        dict(STEP, name="agent_round_x16", layers=8, requests=16, len_lo=12000, len_hi=20000, win_lo=32, win_hi=96,
             keep=0.8, causal=True, tables="fragmented", shape=5),
        # Short actions (a few tokens, "go to shelf 1"): windows of 3-12 tokens, 12-48 window x group rows.
        dict(STEP, name="short_action_x8", layers=12, requests=8, len_lo=6000, len_hi=14000, win_lo=3, win_hi=12,
             keep=0.3, causal=True, tables="fragmented", shape=6),
        # A host program that hands over host buffers: head_dim 64, groups of 8, pages of 32 tokens, ragged lengths.
        dict(STEP, name="host_step_x4", host=True, layers=24, group=8, head_dim=64, page=32, requests=4, len_lo=6000,
             len_hi=16000, win_lo=24, win_hi=64, keep=0.3, causal=True, layers_per_call=8, tables="fragmented", shape=7),
        # One decode step of the streaming mode on all 36 layers: 16 requests with compressed caches of 4K-16K.
        dict(STREAM, name="stream_36_layers_x16", layers=36, requests=16, len_lo=4000, len_hi=16000, shape=8),
        # The same update called layer by layer from the attention hook, two requests: the smallest call of all.
        dict(STREAM, name="stream_1_layer_x2", layers=1, requests=2, len_lo=5000, len_hi=9000, shape=9),
        # The monitor at one decode step: one new logit row per request, 16 requests, some history.
        dict(MONITOR, name="monitor_decode_x16"),
        # An action region ends in the streaming mode: LRFU ranking and in-place compaction of 16 ragged requests.
        dict(REGION, name="region_end_x16", shape=10),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "short", "host", "stream", "stream", "monitor", "region"])
    shape = rng.randrange(1, 1 << 20)
    if kind == "stream":
        lo = _log_uniform(rng, 1000, 16000)
        return dict(STREAM, layers=_log_uniform(rng, 1, 48), kv_heads=rng.choice([4, 8]), group=rng.choice([4, 8]),
                    head_dim=rng.choice([64, 128, 128]), page=rng.choice([16, 16, 32]), requests=_log_uniform(rng, 1, 16),
                    len_lo=lo, len_hi=lo * 2, shape=shape)
    if kind == "monitor":
        rows = rng.choice([1, 1, rng.randrange(2, 9), rng.randrange(32, 97)])
        return dict(MONITOR, requests=_log_uniform(rng, 1, 48), rows_lo=max(1, rows // 2), rows_hi=rows,
                    history=_log_uniform(rng, 70, 3000), vocab=rng.choice([VOCAB, VOCAB, 32003]), shape=shape)
    if kind == "region":
        lo = _log_uniform(rng, 2000, 16000)
        return dict(REGION, layers=rng.randrange(1, 9), kv_heads=rng.choice([4, 8]), requests=_log_uniform(rng, 1, 16),
                    len_lo=lo, len_hi=int(lo * 1.7), keep=rng.uniform(0.2, 0.85), protect=rng.randrange(0, 1200), shape=shape)
    if kind == "host":
        lo = _log_uniform(rng, 2000, 10000)
        return dict(STEP, host=True, layers=rng.randrange(4, 25), kv_heads=rng.choice([4, 8]), group=rng.choice([4, 8]),
                    head_dim=rng.choice([64, 128]), page=rng.choice([16, 32]), requests=_log_uniform(rng, 1, 6), len_lo=lo,
                    len_hi=int(lo * 1.6), win_lo=24, win_hi=rng.randrange(32, 97), keep=rng.uniform(0.2, 0.6), causal=True,
                    layers_per_call=rng.choice([0, 6]), logit_rows=rng.choice([0, 16]), clamp_lo=0.15, clamp_hi=0.4,
                    tables="fragmented", shape=shape)
    # whole steps: about the same number of (token, layer) pairs at every size, 3 K to 1.5 M
    pairs = _log_uniform(rng, 3000, 1500000)
    mean = min(_log_uniform(rng, 1200, 40000), max(1200, pairs))
    requests = max(1, min(32, _log_uniform(rng, 1, max(1, pairs // mean))))
    layers = max(1, min(48, pairs // (mean * requests)))
    case = dict(STEP, layers=layers, kv_heads=rng.choice([4, 8]), group=rng.choice([2, 4, 8, 7]),
                head_dim=rng.choice([64, 128, 128]), page=rng.choice([16, 16, 32, 64]), requests=requests,
                len_lo=int(mean * 0.7), len_hi=int(mean * 1.3), win_lo=32, win_hi=rng.randrange(32, 97),
                keep=rng.uniform(0.15, 0.85), causal=rng.random() < 0.5, lse=rng.choice(["computed", "supplied"]),
                layers_per_call=rng.choice([0, 0, 16]), tables=rng.choice(["permutation", "fragmented"]), shape=shape)
    if kind == "short":
        hi = rng.randrange(1, 15)
        case.update(win_lo=max(1, hi // 4), win_hi=hi, group=rng.choice([2, 4]))
    return case


def _spread(case, lo, hi, salt):
    """One size per request, over the logarithm of [lo, hi]; a matter of the case, not of the seed."""
    rng = random.Random(case["shape"] * 16 + salt)
    return [_log_uniform(rng, lo, hi) if hi > lo else lo for _ in range(case["requests"])]


def _lens(case):
    return _spread(case, case["len_lo"], case["len_hi"], 0)


def _wins(case):
    return _spread(case, case["win_lo"], case["win_hi"], 1)


def _keep(case, lens):
    return [max(1, int(L * case["keep"])) for L in lens]


def _params(case):
    return B.BudgetParams.paper_defaults(int(case["clamp_lo"] * 1e6), int(case["clamp_hi"] * 1e6))


class _Tables:
    """Block tables, lengths and free list as views of one int32 buffer, with a copy to start each pass from."""

    def __init__(self, page_table, seq_len, free_list, free_count):
        parts = [page_table, seq_len, free_list, free_count]
        self.flat = torch.cat([t.reshape(-1) for t in parts])
        self.start = self.flat.clone()
        views, o = [], 0
        for t in parts:
            views.append(self.flat[o:o + t.numel()].view(t.shape))
            o += t.numel()
        self.page_table, self.seq_len, self.free_list, self.free_count = views

    def upload(self):
        self.flat.copy_(self.start)


def _attention_lse(inst):
    """What an attention backend hands over: log sum exp of the scaled logits, float32 [layers, sum_win, q heads]."""
    wl = inst.wl
    NL, Hkv, G, D, P = wl.n_layers, wl.n_kv_heads, wl.group, wl.head_dim, wl.page_size
    out = torch.empty((NL, sum(wl.windows), Hkv * G), dtype=torch.float32, device=inst.pool.device)
    w0 = 0
    for r, (L, W) in enumerate(zip(wl.seq_lens, wl.windows)):
        j = torch.arange(L, device=inst.pool.device)
        slots = inst.page_table[r].long()[j // P] * P + j % P
        for l in range(NL):
            k = inst.pool[l, 0].reshape(-1, Hkv, D)[slots].transpose(0, 1).float()                  # [Hkv, L, D]
            q = inst.q[l, w0:w0 + W].view(W, Hkv, G, D).permute(1, 0, 2, 3).reshape(Hkv, W * G, D).float()
            s = torch.bmm(q, k.transpose(1, 2)) * wl.sm_scale                                       # [Hkv, W G, L]
            if wl.causal:
                last = L - W + torch.arange(W, device=s.device).repeat_interleave(G)
                s.masked_fill_(j[None, None, :] > last[None, :, None], float("-inf"))
            lse = torch.logsumexp(s, dim=-1).view(Hkv, W, G)
            out[l, w0:w0 + W] = lse.permute(1, 0, 2).reshape(W, Hkv * G)
        w0 += W
    return out


def _logits(rows, vocab, seed):
    """Action-token logits, sharpness 0.5 .. 4 per request, falling or rising over the request's rows."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    out = torch.randn((sum(rows), vocab), generator=g, device=DEV)
    sharp = 0.5 + 3.5 * torch.rand(len(rows), generator=g, device=DEV)
    drift = 0.6 * torch.rand(len(rows), generator=g, device=DEV) - 0.3
    n = torch.tensor(rows, device=DEV)
    i = torch.cat([torch.arange(m, device=DEV) / m for m in rows])
    out *= (sharp.repeat_interleave(n) * (1 + drift.repeat_interleave(n) * i))[:, None]
    indptr = torch.zeros(len(rows) + 1, dtype=torch.int32, device=DEV)
    indptr[1:] = torch.cumsum(n, 0)
    return out, indptr


def _prepare_step(case, seed):
    lens, wins = _lens(case), _wins(case)
    keep = _keep(case, lens)
    monitored = case["logit_rows"] > 0
    room = [max(1, int(L * case["clamp_hi"])) for L in lens] if monitored else keep
    wl = synth.Workload("case", case["layers"], case["kv_heads"], case["group"], lens, [min(w, L) for w, L in zip(wins, lens)],
                        room, head_dim=case["head_dim"], page_size=case["page"], causal=case["causal"],
                        table_style=case["tables"], pool_slack=1.05, n_topics=case["topics"], seed=seed)
    inst = synth.generate(wl, DEV)
    tab = _Tables(inst.page_table, inst.seq_len, inst.free_list, inst.free_count)
    comp = H.Compressor(inst.pool, tab.page_table, tab.seq_len, tab.free_list, tab.free_count, wl.n_q_heads, H.sizes_of(inst),
                        layers_per_call=case["layers_per_call"] or None, want_lse=True,
                        lse_layers_per_call=case["layers"])
    comp.sel_idx.zero_()
    comp.score.zero_()
    comp.lse.zero_()
    budget = torch.tensor(keep, dtype=torch.int32, device=DEV)
    logits = indptr = None
    if monitored:
        logits, indptr = _logits([case["logit_rows"]] * case["requests"], VOCAB, seed)
    runner = H.HostStepRunner(comp, inst.q, inst.win_indptr, inst.tok_indptr, budget, wl.sm_scale, wl.causal, logits, indptr,
                              hist_cap=512, params=_params(case) if monitored else None)
    if not case["host"]:
        runner.stage_inputs()
        if case["lse"] == "supplied":
            comp.lse.copy_(_attention_lse(inst))
    # the pages that survivors can go to: all of the pool, or what lies behind the interleaved tables
    first = wl.n_req * inst.page_table.shape[1] if case["tables"] == "interleaved" else 0
    cache = inst.pool.view(torch.int16)[:, :, first:]
    return dict(inst=inst, tab=tab, comp=comp, runner=runner, budget=budget, cache=cache, monitored=monitored,
                supplied=case["lse"] == "supplied", host=case["host"])


def _run_step(s):
    tab, comp, runner = s["tab"], s["comp"], s["runner"]
    if s["host"]:
        out = runner.run()                     # copies the tables and budgets in, synchronises, results on the host
    else:
        tab.upload()
        if s["monitored"]:
            runner.d["bud"].copy_(s["budget"])
            runner.d["hlen"].zero_()
        runner.run_device(lse_supplied=s["supplied"])
        out = {"tables": tab.flat, "bud": runner.d["bud"]}
    return {"out": out, "score": comp.score, "lse": comp.lse, "sel_idx": comp.sel_idx, "keep_indptr": comp.keep_indptr,
            "cache": s["cache"], "status": comp.status, "confidence": runner.d.get("hist")}


def _prepare_stream(case, seed):
    lens = _lens(case)
    R = len(lens)
    wl = synth.Workload("case", case["layers"], case["kv_heads"], case["group"], lens, [1] * R, [max(1, L // 4) for L in lens],
                        head_dim=case["head_dim"], page_size=case["page"], causal=True, table_style="fragmented",
                        pool_slack=1.05, seed=seed)
    inst = synth.generate(wl, DEV)
    comp = H.Compressor(inst.pool, inst.page_table, inst.seq_len, inst.free_list, inst.free_count, wl.n_q_heads,
                        H.sizes_of(inst))
    g = torch.Generator(device=DEV)
    g.manual_seed(seed + 1)
    comp.score.copy_(torch.rand(comp.score.shape, generator=g, device=DEV) / max(lens))
    steps = torch.full((R,), 3, dtype=torch.int32, device=DEV)
    return dict(inst=inst, comp=comp, lse=_attention_lse(inst), steps=steps)


def _run_stream(s):
    inst, comp, sz = s["inst"], s["comp"], s["comp"].sz
    B.actkv_score_accumulate(comp.pd, comp.td, 0, inst.wl.n_layers, inst.q, inst.win_indptr, inst.wl.n_q_heads, s["lse"],
                             inst.wl.sm_scale, True, inst.tok_indptr, s["steps"], comp.score, sz.sum_win, sz.max_win,
                             sz.sum_tok, sz.max_tok, comp.ws_score, comp.status)
    return {"score": comp.score, "status": comp.status}


def _rows(case):
    return _spread(case, case["rows_lo"], case["rows_hi"], 2)


def _prepare_monitor(case, seed):
    rows = _rows(case)
    R, n_rows = len(rows), sum(rows)
    logits, indptr = _logits(rows, case["vocab"], seed)
    cap = case["history"] + 128
    g = torch.Generator(device=DEV)
    g.manual_seed(seed + 1)
    i = torch.arange(cap, device=DEV) / cap
    hist = (4.0 + torch.rand((R, 1), generator=g, device=DEV) * i + 0.5 * torch.rand((R, cap), generator=g, device=DEV))
    length = torch.full((R,), case["history"], dtype=torch.int32, device=DEV)
    i32 = lambda v: torch.full((R,), v, dtype=torch.int32, device=DEV)  # noqa: E731
    ws = torch.empty(B.actkv_budget_workspace_bytes(n_rows, R, cap) + 256, dtype=torch.uint8, device=DEV)
    return dict(logits=logits, indptr=indptr, n_rows=n_rows, vocab=case["vocab"], hist=hist.contiguous(), cap=cap, R=R,
                length0=length, length=length.clone(), params=B.BudgetParams.paper_defaults(), budget=i32(2048),
                budget_out=i32(0), slope=torch.zeros(R, dtype=torch.float64, device=DEV), ws=ws, status=torch.zeros(4, dtype=torch.int32, device=DEV))


def _run_monitor(s):
    s["length"].copy_(s["length0"])            # every pass appends to the same history
    B.actkv_budget(s["logits"], s["indptr"], s["n_rows"], s["vocab"], s["hist"], s["length"], s["cap"], s["params"], None,
                   s["budget"], s["budget_out"], s["slope"], s["R"], s["ws"], s["status"])
    return {"confidence": s["hist"], "length": s["length"], "budget": s["budget_out"], "slope": s["slope"],
            "status": s["status"]}


def _prepare_region(case, seed):
    lens = _lens(case)
    wl = synth.Workload("case", case["layers"], case["kv_heads"], case["group"], lens, [1] * len(lens), _keep(case, lens),
                        head_dim=case["head_dim"], page_size=case["page"], causal=True, table_style="fragmented",
                        pool_slack=1.05, seed=seed)
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    g_cpu = torch.Generator()
    g_cpu.manual_seed(seed)
    table, seq_len, free_list, free_count, n_pages = synth.make_tables(wl, DEV, g_cpu)
    pool = torch.empty((wl.n_layers, 2, n_pages, wl.page_size, wl.n_kv_heads, wl.head_dim), dtype=torch.bfloat16, device=DEV)
    pool.normal_(generator=g)
    tab = _Tables(table, seq_len, free_list, free_count)
    sizes = H.StepSizes(wl.n_req, wl.n_req, 1, sum(lens), max(lens), sum(wl.budgets), max(wl.budgets))
    comp = H.Compressor(pool, tab.page_table, tab.seq_len, tab.free_list, tab.free_count, wl.n_q_heads, sizes)
    # pooled attention mass: log-normal around 1 / L, two percent of the entries strongly attended
    n_outer = wl.n_layers * wl.n_kv_heads
    x = torch.exp(torch.randn((n_outer, sizes.sum_tok), generator=g, device=DEV)) / max(lens)
    x *= torch.where(torch.rand(x.shape, generator=g, device=DEV) < 0.02, 20.0, 1.0)
    comp.score.view(n_outer, -1).copy_(x.clamp_(max=1.0))
    comp.sel_idx.zero_()
    protect = torch.tensor([min(case["protect"], L) for L in lens], dtype=torch.int32, device=DEV)
    lrfu = H.LrfuState(n_outer, sizes, DEV, top_p=0.9, lam=0.5, n_protect=protect)
    # two thirds of the entries were there before this round and carry a keep-score
    old = torch.exp(torch.randn(x.shape, generator=g, device=DEV)) / max(lens)
    lrfu.keep_score.copy_(torch.where(torch.rand(x.shape, generator=g, device=DEV) < 0.66, old, 0.0))
    tok = torch.zeros(len(lens) + 1, dtype=torch.int32)
    tok[1:] = torch.cumsum(torch.tensor(lens), 0)
    budget = torch.tensor(wl.budgets, dtype=torch.int32, device=DEV)
    comp.new_order = torch.zeros_like(comp.sel_idx)
    return dict(comp=comp, tab=tab, lrfu=lrfu, tok=tok.to(DEV), budget=budget, cache=pool.view(torch.int16), layers=wl.n_layers)


def _run_region(s):
    comp, lrfu, tab, NL = s["comp"], s["lrfu"], s["tab"], s["layers"]
    tab.upload()
    B.actkv_keep_indptr(comp.seq_len, s["budget"], comp.sz.n_req, comp.keep_indptr)
    comp.run_keepscore_select(lrfu, s["tok"], s["budget"], 0, NL)
    comp.run_compact_inplace(s["budget"], 0, NL)
    comp.run_gather_ks(lrfu, s["tok"], 0, NL, idx=comp.new_order)
    return {"keep_score": lrfu.keep_score, "kept": lrfu.kept, "sel_idx": comp.sel_idx, "order": comp.new_order,
            "tables": tab.flat, "cache": s["cache"], "status": comp.status}


def prepare(case, seed):
    kind = case["kind"]
    made = {"step": _prepare_step, "stream": _prepare_stream, "monitor": _prepare_monitor, "region": _prepare_region}[kind](case, seed)
    return dict(made, kind=kind)


def run(state):
    return {"step": _run_step, "stream": _run_stream, "monitor": _run_monitor, "region": _run_region}[state["kind"]](state)


def work(case):
    """Bytes that have to be read or written once, operations of the contractions that have to be made once."""
    if case["kind"] == "monitor":
        return {"bytes": 4.0 * sum(_rows(case)) * case["vocab"], "flops": 4.0 * sum(_rows(case)) * case["vocab"]}
    lens = _lens(case)
    D, units = case["head_dim"], case["layers"] * case["kv_heads"]
    if case["kind"] == "stream":
        return {"bytes": float(units * sum(lens) * (2 * D + 8)), "flops": float(units * sum(lens) * 2 * D * case["group"])}
    keep = _keep(case, lens)
    if case["kind"] == "region":
        # scores read, keep-scores read and written; kept: index, order, gathered keep-score (read, written); a kept
        # row outside the tail region (a share 1 - B / L of them) is read and written, K and V
        moved = sum(n * (1.0 - n / L) for n, L in zip(keep, lens))
        return {"bytes": units * (12.0 * sum(lens) + 16.0 * sum(keep) + 8.0 * D * moved), "flops": 0.0}
    rows = [w * case["group"] for w in _wins(case)]
    # K rows read, scores written; survivors: index, V row read, K and V row written; logits; host: queries cross the link
    byts = units * ((2.0 * D + 4) * sum(lens) + (6.0 * D + 4) * sum(keep)) + 4.0 * case["logit_rows"] * case["requests"] * VOCAB
    byts += case["layers"] * case["kv_heads"] * sum(rows) * 2.0 * D
    return {"bytes": byts, "flops": 2.0 * D * units * sum(n * L for n, L in zip(rows, lens))}


def tolerance(case):
    # Scores and LSE are float32 sums of up to 64K exponentials of float32 dot products of bf16 numbers: measured against
    # float64 on five shapes, relative error 1.4e-7 to 4.8e-7 (2-norm) and 1.4e-6 (largest).  Two entries
    # whose scores agree to the last bits may change places at the budget's threshold; every later survivor of that
    # (layer, head, request) then sits one slot further, so whole numbers (indices, cache bytes) carry a small share.
    if case["kind"] == "step":
        return {"rel": 5e-6, "max": 5e-5, "differ": 0.01}
    if case["kind"] == "stream":
        return {"rel": 5e-6, "max": 5e-5}
    if case["kind"] == "monitor":
        return {"rel": 1e-5, "max": 1e-4}
    return "exact"                              # one rounding per operation is part of the keep-score's definition
