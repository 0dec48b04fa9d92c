"""Decode steps of the packed-wavefront library, sized as its users run it.

A case is one decode step of a batch: pack the live blocks, run the attention of
``layers`` layers over them, turn the last hidden states or logits into token
decisions, commit and admit.  Shapes come from the benchmark workloads and the
parity workloads of this repository (request counts 1 to 128, blocks of 32 to
128 tokens, windows of 2 to 5 blocks, prefixes of tens to tens of thousands of
tokens, three head layouts, 1,024 to 151,552 tokens of vocabulary); ``draw``
spreads over the same ranges.

  kv      "window": the step's K/V stay in slot order and are copied to the pages
                    when a block retires
          "pages":  they are scattered to the pages every step (rotary embedding
                    applied on the way), the attention reads pages only
          "fp8":    the same with 8-bit (E4M3) pages
  head    "logits": the row pass reads bf16 logits; "lm_head": it is fused into
          the head's matrix product and takes hidden states of size ``hidden``
  moves   False: no confidence reaches a threshold, so the state stays as it is
          (most forwards of most requests, and the plain throughput of a step);
          True: tokens are revealed and edited, blocks retire and are admitted.
          The scheduler then writes the rows of its requests before the step (one
          copy), so every pass starts from the same state
  sync    the batch-synchronous commit and admission rule
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2607_17652_b200 import binding as B

DEV = "cuda"
PAGE = 64
THRESHOLDS = (0.9, 0.95)          # tau_mask, tau_edit
ROPE_BASE = 10000.0


def _case(name, requests, block_len, wmax, prefix, live, heads, vocab, **more):
    q_heads, kv_heads, head_dim = heads
    c = dict(name=name, requests=requests, block_len=block_len, wmax=wmax, prefix_lo=prefix[0], prefix_hi=prefix[1],
             live_lo=live[0], live_hi=live[1], q_heads=q_heads, kv_heads=kv_heads, head_dim=head_dim, vocab=vocab,
             layers=1, kv="window", head="logits", hidden=0, moves=False, sync=False)
    c.update(more)
    return c


SMALL, MEDIUM, LARGE = (4, 1, 64), (16, 4, 128), (32, 8, 128)
V_LLM = 151552


def listed():
    return [
        # one request of a toy model: nothing but launch latency and short dependent chains
        _case("single_tiny", 1, 32, 2, (64, 64), (2, 2), SMALL, 1024),
        # batch size 1, the latency-critical setting: one user, a few thousand tokens of context,
        # the attention of several layers of a full-size model per step
        _case("single_chat", 1, 32, 2, (3001, 3001), (2, 2), LARGE, V_LLM, layers=4, kv="pages"),
        # batch size 1 with a long document in the prefix
        _case("single_document", 1, 32, 4, (28123, 28123), (3, 3), LARGE, V_LLM, moves=True),
        # a small batch on a medium model
        _case("batch8", 8, 32, 4, (256, 2048), (1, 4), MEDIUM, V_LLM),
        # the same batch as an engine runs it: all pages, several layers, blocks that commit
        _case("batch8_layers", 8, 32, 4, (256, 2048), (1, 4), MEDIUM, V_LLM, layers=4, kv="pages", moves=True),
        # a middling batch under the batch-synchronous rule, longer blocks
        _case("batch24_sync", 24, 64, 3, (700, 5000), (1, 3), LARGE, V_LLM, moves=True, sync=True),
        # the serving batch
        _case("batch64", 64, 32, 4, (1024, 8192), (1, 4), LARGE, V_LLM),
        # ... with the cache held in 8 bits
        _case("batch64_fp8", 64, 32, 4, (1024, 8192), (1, 4), LARGE, V_LLM, kv="fp8", moves=True),
        # ... with the row pass fused into the head's matrix product
        _case("batch64_head", 64, 32, 4, (1024, 8192), (1, 4), LARGE, V_LLM, head="lm_head", hidden=2048, moves=True),
        # long contexts
        _case("long16", 16, 64, 3, (16384, 32768), (3, 3), LARGE, V_LLM),
        # ... in 8 bits
        _case("long16_fp8", 16, 64, 3, (16384, 32768), (3, 3), LARGE, V_LLM, kv="fp8"),
        # the widest batch: short and middling prefixes, blocks that commit, all pages
        _case("serving128", 128, 32, 4, (512, 4096), (1, 4), LARGE, V_LLM, kv="pages", moves=True),
    ]


def draw(rng):
    log = lambda lo, hi: math.exp(rng.uniform(math.log(lo), math.log(hi)))
    q_heads, kv_heads, head_dim = rng.choice(
        [SMALL, (8, 2, 64), MEDIUM, MEDIUM, LARGE, LARGE, LARGE, (12, 3, 128), (16, 2, 128), (4, 4, 128)])
    group = q_heads // kv_heads
    block_len = rng.choice([b for b in (32, 32, 64, 96, 128) if b * group % 128 == 0])
    wmax = rng.randint(2, 5 if block_len <= 64 else 3)
    live_lo = rng.randint(1, wmax)
    live_hi = rng.randint(live_lo, wmax)
    requests = round(log(1, 128))
    prefix_hi = round(log(48, 32768))
    prefix_lo = round(prefix_hi * rng.uniform(0.1, 1.0))
    vocab = rng.choice([V_LLM, V_LLM, 8 * round(log(1024, V_LLM) / 8)])
    kv = rng.choice(["window", "pages", "fp8"] if head_dim == 128 else ["window", "pages"])
    head = rng.choice(["logits", "logits", "logits", "lm_head"])
    # (retiring a block freezes one layer's K/V where the window is kept in slot order)
    c = _case("", requests, block_len, wmax, (prefix_lo, prefix_hi), (live_lo, live_hi), (q_heads, kv_heads, head_dim),
              vocab, layers=rng.choice([1, 1, 2, 4]) if kv != "window" else 1, kv=kv, head=head,
              hidden=64 * round(log(512, 4096) / 64) if head == "lm_head" else 0,
              moves=rng.random() < 0.6, sync=rng.random() < 0.2)
    del c["name"]
    # no dearer than the dearest of the list
    limit = max(_cost(k) for k in listed())
    while c["requests"] > 1 and (_cost(c) > limit or c["requests"] * wmax * block_len * vocab > 2.5e9):
        c["requests"] = c["requests"] * 3 // 4
    while _cost(c) > limit:
        c["prefix_hi"], c["prefix_lo"] = c["prefix_hi"] // 2, c["prefix_lo"] // 2
    return c


def _cost(case):
    """Seconds, roughly: operations at 1e15 (attention) and 1.4e15 (head) a second, bytes at 6e12."""
    w, without = work(case), work(dict(case, head="logits"))
    return without["flops"] / 1.0e15 + (w["flops"] - without["flops"]) / 1.4e15 + w["bytes"] / 6e12


def work(case):
    """Expected bytes and operations of a step.  Attention: K and V of what a request sees once
    per KV head, Q once, the output once, two products over the visible pairs.  Row pass: the
    logits of the live rows once; with the fused head, its weights once and the product."""
    n, b = case["requests"], case["block_len"]
    p = (case["prefix_lo"] + case["prefix_hi"]) / 2
    ws = range(case["live_lo"], case["live_hi"] + 1)
    w = sum(ws) / len(ws)
    pairs = n * sum(sum(b * (p + (s + 1) * b) for s in range(k)) for k in ws) / len(ws)
    rows = n * w * b
    d, hq, hkv = case["head_dim"], case["q_heads"], case["kv_heads"]
    cache = 1 if case["kv"] == "fp8" else 2
    layer = n * (p + w * b) * 2 * hkv * d * cache + rows * 2 * hq * d * 2
    if case["kv"] != "window":                       # fresh K/V in (the pages they go to are counted above)
        layer += rows * 2 * hkv * d * 2
    flops = case["layers"] * 4.0 * d * hq * pairs
    if case["head"] == "logits":
        head = rows * case["vocab"] * 2
    else:
        head = case["vocab"] * case["hidden"] * 2 + rows * case["hidden"] * 2
        flops += 2.0 * rows * case["vocab"] * case["hidden"]
    return {"bytes": case["layers"] * layer + head + rows * 25, "flops": flops}


def tolerance(case):
    """bf16 attention against the fp64 oracle: 2.2e-3 to 2.4e-3 in the 2-norm at every size (bf16
    weights and outputs).  With 8-bit pages the kernel rounds queries and weights to E4M3 (three
    mantissa bits): 3.6e-2 against exact arithmetic, so 3e-2 between two kernels that do.  Token
    ids, decisions and state are whole numbers and the same; only the fused head sums its
    logits in fp32 in an order of its own, so that near-equal candidates may change places, and
    a rotated key may fall on the other side of an 8-bit rounding step."""
    t = {"rel": 3e-2 if case["kv"] == "fp8" else 1e-2, "max": 0.99 if case["kv"] == "fp8" else 0.4}
    if case["head"] == "lm_head":
        t["differ"] = 1e-3
    elif case["kv"] == "fp8":
        t["differ"] = 1e-4
    return t


# ------------------------------------------------------------------ inputs
def _structure(case, rng):
    """Prefix lengths and live-block counts, one draw from each of ``requests`` equal slices of
    their ranges (so that two seeds ask for nearly the same work), and a page table that scatters
    the pages of all requests over one pool."""
    n, b, wmax = case["requests"], case["block_len"], case["wmax"]
    u = (np.arange(n) + rng.random(n)) / n
    prefix = case["prefix_lo"] + np.floor(u * (case["prefix_hi"] - case["prefix_lo"] + 1)).astype(np.int64)
    u = (np.arange(n) + rng.random(n)) / n
    live = case["live_lo"] + np.floor(u * (case["live_hi"] - case["live_lo"] + 1)).astype(np.int64)
    prefix, live = rng.permutation(prefix), rng.permutation(live)
    blocks = 32
    left = np.minimum(np.minimum(prefix // b, rng.integers(0, 9, n)), blocks - wmax)
    need = -(-(prefix + wmax * b) // PAGE)
    # the pool and the table are sized for the longest prefix of every slice: the same for every seed
    top = case["prefix_lo"] + np.floor(np.arange(1, n + 1) / n * (case["prefix_hi"] - case["prefix_lo"] + 1))
    most = -(-(top.astype(np.int64) + wmax * b) // PAGE)
    table = np.zeros((n, int(most.max())), np.int32)
    pages = int(most.sum())
    perm, at = rng.permutation(pages), 0
    for r in range(n):
        table[r] = perm[at]
        table[r, :need[r]] = perm[at:at + need[r]]
        at += need[r]
    return prefix, left, left + live, table, pages, blocks


def _tokens(case, rng, left, right, blocks):
    """Live blocks: a share of [M] drawn per block (one at least, so that nothing is finished
    before the step), token ids elsewhere; everything to the right is [M]."""
    n, b, V = case["requests"], case["block_len"], case["vocab"]
    tok = rng.integers(0, V - 2, (n, blocks, b)).astype(np.int32)
    for r in range(n):
        for g in range(left[r], right[r]):
            masks = b // 2 if not case["moves"] else max(1, round(rng.random() ** 2 * b))
            tok[r, g, rng.permutation(b)[:masks]] = V - 1
        tok[r, right[r]:] = V - 1
    return tok.reshape(n, blocks * b)


def _confidences(case, rng, rows):
    """Target confidence and winner of each live row: 85 % get one, away from both thresholds by
    more than any rounding moves them."""
    c = np.clip(rng.uniform(0.5, 1.35, rows), 0.0, 0.99)
    for t in THRESHOLDS:
        near = np.abs(c - t) < 8e-3
        c[near] = t + 1.2e-2
    return c, rng.integers(0, case["vocab"] - 2, rows), rng.random(rows) < 0.85


def _randn(shape, gen, std=1.0):
    x = torch.randn(shape, device=DEV, dtype=torch.bfloat16, generator=gen)
    return x.mul_(std) if std != 1.0 else x


def _row_statistics(z, winners):
    """log of the sum of exponentials over all columns but the winner's, in row slices."""
    out = []
    for at in range(0, z.shape[0], 1024):
        x = z[at:at + 1024].float()
        x.scatter_(1, winners[at:at + 1024, None], -math.inf)
        out.append(torch.logsumexp(x, 1))
    return torch.cat(out)


def _logits(case, gen, conf, winners, picked, rows, total):
    """N(0, 1) logits of the live rows; the winner's is set so that its softmax confidence comes
    out as asked, or, where nothing moves, raised by 6 on 70 % of the rows (which a vocabulary of
    this size leaves far below every threshold).  [M] and EOS never win."""
    z = torch.zeros((total, case["vocab"]), device=DEV, dtype=torch.bfloat16)
    z[:rows].normal_(generator=gen)
    z[:, -2:] = -10.0
    win = torch.from_numpy(winners).to(DEV)
    at = torch.arange(rows, device=DEV)
    if case["moves"]:
        p = torch.from_numpy(conf).to(DEV)
        a = (torch.log(p / (1 - p)) + _row_statistics(z[:rows], win)).to(torch.bfloat16)
        z[at, win] = torch.where(torch.from_numpy(picked).to(DEV), a, z[at, win])
    elif case["vocab"] >= 8192:
        z[at, win] += torch.from_numpy(np.where(np.arange(rows) % 10 < 7, 6.0, 0.0)).to(DEV, torch.bfloat16)
    return z


def _hidden(case, gen, conf, winners, picked, rows, total):
    """Hidden states and head weights whose logits look like those of ``_logits``: a row is moved
    along its winner's weight vector until the confidence is as asked."""
    h, V = case["hidden"], case["vocab"]
    w = _randn((V, h), gen, 1.0 / math.sqrt(h))
    w[-2:] = 0
    x = torch.zeros((total, h), device=DEV, dtype=torch.bfloat16)
    x[:rows].normal_(generator=gen)
    if case["moves"]:
        p, pick = torch.from_numpy(conf).to(DEV), torch.from_numpy(picked).to(DEV)
        win = torch.from_numpy(winners).to(DEV)
        for at in range(0, rows, 2048):
            s = slice(at, min(at + 2048, rows))
            wv = w[win[s]].float()
            goal = x[s].float()
            for _ in range(2):                       # the rounded row moves the other logits a little: once more
                z = goal.to(torch.bfloat16) @ w.T
                rest = _row_statistics(z, win[s])
                have = (goal.to(torch.bfloat16).float() * wv).sum(1)
                want = torch.log(p[s] / (1 - p[s])).float() + rest
                goal = goal + ((want - have) / (wv * wv).sum(1))[:, None] * wv
            x[s] = torch.where(pick[s, None], goal.to(torch.bfloat16), x[s])
    return x, w


class _State:
    pass


def prepare(case, seed):
    rng = np.random.Generator(np.random.Philox(key=[seed & 0xFFFFFFFF, 21]))
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    n, b, V = case["requests"], case["block_len"], case["vocab"]
    prefix, left, right, table, pages, blocks = _structure(case, rng)
    tokens = _tokens(case, rng, left, right, blocks)
    rows, total = int((right - left).sum()) * b, n * case["wmax"] * b
    conf, winners, picked = _confidences(case, rng, rows)
    # a revealed position mostly holds its winner already; the others are the ones edits go for
    r = np.repeat(np.arange(n), (right - left) * b)
    col = np.concatenate([np.arange(lo * b, hi * b) for lo, hi in zip(left, right)])
    keep = (tokens[r, col] != V - 1) & (rng.random(rows) < 0.9)
    tokens[r[keep], col[keep]] = winners[keep]

    s = _State()
    s.case = case
    s.ctx = B.Context(max_requests=n, wmax=case["wmax"], block_len=b, n_q_heads=case["q_heads"],
                      n_kv_heads=case["kv_heads"], head_dim=case["head_dim"], page_size=PAGE, num_pages=pages,
                      max_pages_per_req=table.shape[1], vocab=V, mask_id=V - 1, eos_id=V - 2, max_blocks=blocks,
                      s_pe=0 if case["moves"] else 1, tau_mask=THRESHOLDS[0], tau_edit=THRESHOLDS[1], theta_spawn=0.5,
                      sm_scale=0.0, window_in_pages=int(case["kv"] != "window"), batch_sync=int(case["sync"]),
                      kv_fp8=int(case["kv"] == "fp8"))
    # the scheduler's rows in one buffer, so that it can write them with one copy
    pad = lambda k: -(-k // 64) * 64
    parts = [np.ones(n), prefix, left, right, tokens]
    sizes = [pad(p.size) for p in parts] + [pad(n * case["wmax"])]
    rows0 = np.zeros(sum(sizes), np.int32)
    at, views = 0, []
    s.rows = torch.empty(rows0.size, dtype=torch.int32, device=DEV)
    for p, size in zip(parts, sizes):
        rows0[at:at + p.size] = np.asarray(p).reshape(-1)
        views.append(s.rows[at:at + p.size].view(p.shape))
        at += size
    pe = s.rows[at:].view(torch.uint8)[:n * case["wmax"]].view(n, case["wmax"])
    s.rows0 = torch.from_numpy(rows0).to(DEV)
    s.rows.copy_(s.rows0)
    s.st = B.DeviceState(*views, pe, torch.from_numpy(table).to(DEV))

    s.pk = B.PackBuffers.alloc(s.ctx, DEV)
    s.sb = B.StepBuffers(s.ctx, DEV)
    hq, hkv, d = case["q_heads"], case["kv_heads"], case["head_dim"]
    s.layers = []
    for i in range(case["layers"]):
        lay = {"q": _randn((total, hq, d), gen), "k_new": _randn((total, hkv, d), gen),
               "v_new": _randn((total, hkv, d), gen)}
        shape = (pages, hkv, PAGE, d)
        if case["kv"] == "fp8":
            for name in ("k", "v"):
                scale = 6.0 / 448.0 * (0.5 + 1.5 * torch.rand(hkv, device=DEV, generator=gen))
                pool = torch.empty(shape, dtype=torch.uint8, device=DEV)
                for p0 in range(0, pages, 4096):
                    x = torch.randn(pool[p0:p0 + 4096].shape, device=DEV, generator=gen) / scale[None, :, None, None]
                    pool[p0:p0 + 4096] = x.clamp_(-448.0, 448.0).to(torch.float8_e4m3fn).view(torch.uint8)
                lay[name + "_scale"], lay[name + "_pool"] = scale, pool
        else:
            lay["k_pool"], lay["v_pool"] = _randn(shape, gen), _randn(shape, gen)
        lay["out"] = s.sb.out if i == 0 else torch.zeros_like(s.sb.out)
        s.layers.append(lay)
    if case["head"] == "logits":
        s.logits = _logits(case, gen, conf, winners, picked, rows, total)
    else:
        s.x, s.w = _hidden(case, gen, conf, winners, picked, rows, total)
        s.head_ws = torch.zeros(B.lib().fb_lm_head_workspace_bytes(s.ctx.handle), dtype=torch.uint8, device=DEV)
    return s


# ---------------------------------------------------------------- one step
def run(s):
    case, ctx, st, pk, sb = s.case, s.ctx, s.st, s.pk, s.sb
    if case["moves"]:
        s.rows.copy_(s.rows0)                        # the scheduler writes the rows of its requests
    B.fb_pack_wavefronts(ctx, st, pk, sb.ws, sb.status)
    for a in s.layers:
        if case["kv"] == "window":
            B.fb_wavefront_attn(ctx, pk, a["q"], a["k_new"], a["v_new"], a["k_pool"], a["v_pool"], st.page_table,
                                a["out"], sb.ws, sb.status)
        elif case["kv"] == "pages":
            B.fb_scatter_window_kv(ctx, pk, st.page_table, a["k_new"], a["v_new"], a["k_pool"], a["v_pool"], sb.status,
                                   ROPE_BASE)
            B.fb_wavefront_attn(ctx, pk, a["q"], None, None, a["k_pool"], a["v_pool"], st.page_table, a["out"], sb.ws,
                                sb.status)
        else:
            B.fb_scatter_window_kv_fp8(ctx, pk, st.page_table, a["k_new"], a["v_new"], a["k_pool"], a["v_pool"],
                                       a["k_scale"], a["v_scale"], sb.status, ROPE_BASE)
            B.fb_wavefront_attn_fp8(ctx, pk, a["q"], a["k_pool"], a["v_pool"], a["k_scale"], a["v_scale"],
                                    st.page_table, a["out"], sb.ws, sb.status)
    if case["head"] == "logits":
        B.fb_t2t_step(ctx, pk, s.logits, st, sb.argmax, sb.conf, sb.action, sb.slot_stats, sb.status)
    else:
        B.fb_lm_head_t2t(ctx, pk, s.x, s.w, st, sb.argmax, sb.conf, sb.action, sb.slot_stats, s.head_ws, sb.status)
    # (the pages of every layer already hold the window, or there is one layer)
    win = case["kv"] == "window"
    a = s.layers[-1]
    B.fb_gate_commit(ctx, pk, sb.slot_stats, st, a["k_new"] if win else None, a["v_new"] if win else None, a["k_pool"],
                     a["v_pool"], sb.n_committed, sb.spawned, sb.step_counters, sb.status)
    return {"out": [a["out"] for a in s.layers], "k_pool": [a["k_pool"] for a in s.layers],
            "v_pool": [a["v_pool"] for a in s.layers], "qtok": pk.qtok, "pos": pk.pos, "slot_req": pk.slot_req,
            "slot_s": pk.slot_s, "slot_pos0": pk.slot_pos0, "slot_kv_len": pk.slot_kv_len, "slot_flags": pk.slot_flags,
            "req_slot_begin": pk.req_slot_begin, "n_live": pk.n_live, "argmax": sb.argmax, "conf": sb.conf,
            "action": sb.action, "slot_stats": sb.slot_stats, "n_committed": sb.n_committed, "spawned": sb.spawned,
            "counters": sb.step_counters, "status": sb.status, "active": st.active, "prefix_len": st.prefix_len,
            "L": st.L, "R": st.R, "tokens": st.tokens, "pe_done": st.pe_done}
