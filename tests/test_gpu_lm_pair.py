"""The LM head with two CTAs to a tile: row tiles in even and odd numbers (one CTA, pairs, pairs with an idle
half), ragged last row and vocabulary tiles, winners on both sides of a pair's division of W."""
import numpy as np
import pytest
import torch

from oracle import flowblock_oracle as O
from paper_2607_17652_b200 import binding as B
from paper_2607_17652_b200 import synth
from tests import harness as H

DEV = "cuda:0"
pytestmark = pytest.mark.gpu
V, HIDDEN, BL, REQUESTS, WMAX = 296 * 256 + 8, 768, 32, 16, 4     # 297 vocabulary tiles, 16 row tiles of capacity


@pytest.fixture(scope="module")
def head():
    rg = np.random.default_rng(5)
    rows = REQUESTS * WMAX * BL
    w = synth.randn_bf16((V, HIDDEN), 41, 13, 1.0 / np.sqrt(HIDDEN))
    x = synth.randn_bf16((rows, HIDDEN), 41, 14)
    # a clear winner in every 16th row, at the edges of the vocabulary tiles and of their halves among others
    edges = [0, 127, 128, 255, 256, V - 9, V - 8, V - 3]
    winners = {r: edges[i % 16] if i % 16 < len(edges) else int(rg.integers(0, V - 2)) for i, r in enumerate(range(0, rows, 16))}
    for r, wi in winners.items():
        wv = w[wi].to(torch.float64)
        x[r] = (x[r].to(torch.float64) + rg.uniform(12.0, 15.0) * wv / float(wv @ wv)).to(torch.bfloat16)
    return x, w, winners


# live blocks (row tiles): 4 (1), 8 (2), 9 (3, ragged), 13 (4, ragged), 49 (13, ragged), 64 (16)
@pytest.mark.parametrize("blocks", [4, 8, 9, 13, 49, 64])
def test_lm_head_row_tiles_in_pairs(head, blocks):
    x, w, winners = head
    live = np.array([min(WMAX, max(0, blocks - WMAX * r)) for r in range(REQUESTS)], np.int32)
    ctx = B.Context(max_requests=REQUESTS, wmax=WMAX, block_len=BL, n_q_heads=4, n_kv_heads=1, head_dim=64, page_size=64,
                    num_pages=8, max_pages_per_req=4, vocab=V, mask_id=V - 1, eos_id=V - 2, max_blocks=8, s_pe=1,
                    tau_mask=0.9, tau_edit=0.95, theta_spawn=0.5, sm_scale=0.0)
    st = B.DeviceState.from_numpy(DEV, np.ones(REQUESTS, np.int32), np.zeros(REQUESTS, np.int32), np.zeros(REQUESTS, np.int32),
                                  live, np.zeros((REQUESTS, 8 * BL), np.int32), np.zeros((REQUESTS, WMAX), np.uint8),
                                  np.zeros((REQUESTS, 4), np.int32))
    pk, sb = B.PackBuffers.alloc(ctx, DEV), B.StepBuffers(ctx, DEV)
    ws = torch.zeros(B.lib().fb_lm_head_workspace_bytes(ctx.handle), dtype=torch.uint8, device=DEV)
    B.fb_pack_wavefronts(ctx, st, pk, sb.ws, sb.status)
    B.fb_lm_head_t2t(ctx, pk, x.to(DEV), w.to(DEV), st, sb.argmax, sb.conf, sb.action, sb.slot_stats, ws, sb.status)
    torch.cuda.synchronize()
    assert int(sb.status.item()) == 0
    rows = blocks * BL
    # the oracle's row pass over the sampled rows, packed as the blocks of a small problem of their own
    sample = [r for r in winners if r < rows]
    sample = sample[:16] + sample[-16:] if len(sample) > 32 else sample
    mstc = synth.make_structure(synth.tiny_workload(n_requests=1, wmax=1, w_lo=1, w_hi=1, prefix_lo=0, prefix_hi=0, vocab=V))
    mcfg = H.oracle_cfg(mstc)
    mpk = O.pack_wavefronts(mcfg, H.oracle_state(mstc, synth.make_tokens(mstc)))
    assert mpk.n_live * mcfg.block_len == 32
    z = np.zeros((mcfg.max_slots * mcfg.block_len, V))
    xs = H.f64(x[torch.tensor(sample)])
    for v0 in range(0, V, 16384):
        z[:len(sample), v0:v0 + 16384] = xs @ H.f64(w[v0:v0 + 16384]).T
    xo, co = O.t2t_rows(mcfg, mpk, z)
    np.testing.assert_array_equal(sb.argmax.cpu().numpy()[sample], xo[:len(sample)])
    np.testing.assert_array_equal(xo[:len(sample)], [winners[r] for r in sample])
    # fp32 accumulation of 768 products of a few units against fp64: |dz| < 1e-4, dp <= p (1 - p) |dz| and the
    # sum's own rounding
    err = np.abs(sb.conf.cpu().numpy()[sample] - co[:len(sample)])
    assert err.max() <= 1e-4, err.max()
    am, cf = sb.argmax.cpu().numpy(), sb.conf.cpu().numpy()
    assert ((am[:rows] >= 0) & (am[:rows] < V)).all() and ((cf[:rows] > 0) & (cf[:rows] <= 1)).all()
    assert (am[rows:] == -1).all() and not cf[rows:].any()


# ---- all rows, bit for bit, against the one-CTA form (which form runs where: test_lm_forms.py)
class Head:
    def __init__(self, requests, vocab):
        self.ctx = B.Context(max_requests=requests, wmax=WMAX, block_len=BL, n_q_heads=4, n_kv_heads=1, head_dim=64, page_size=64,
                             num_pages=8, max_pages_per_req=4, vocab=vocab, mask_id=vocab - 1, eos_id=vocab - 2, max_blocks=8, s_pe=1,
                             tau_mask=0.9, tau_edit=0.95, theta_spawn=0.5, sm_scale=0.0)
        self.requests, self.rows = requests, requests * WMAX * BL
        self.ws = torch.zeros(B.lib().fb_lm_head_workspace_bytes(self.ctx.handle), dtype=torch.uint8, device=DEV)

    def run(self, x, w, blocks):
        """`x`: as many rows as the context holds.  (argmax, conf, status, action, state)"""
        live = np.array([min(WMAX, max(0, blocks - WMAX * r)) for r in range(self.requests)], np.int32)
        n, z = self.requests, np.zeros
        tokens = np.full((n, 8 * BL), self.ctx.cfg.mask_id, np.int32)
        st = B.DeviceState.from_numpy(DEV, np.ones(n, np.int32), z(n, np.int32), z(n, np.int32), live, tokens,
                                      z((n, WMAX), np.uint8), z((n, 4), np.int32))
        pk, sb = B.PackBuffers.alloc(self.ctx, DEV), B.StepBuffers(self.ctx, DEV)
        B.fb_pack_wavefronts(self.ctx, st, pk, sb.ws, sb.status)
        B.fb_lm_head_t2t(self.ctx, pk, x, w, st, sb.argmax, sb.conf, sb.action, sb.slot_stats, self.ws, sb.status)
        torch.cuda.synchronize()
        return sb.argmax, sb.conf, int(sb.status.item()), sb.action, st


def one_cta(x, w, blocks):
    """The same rows three row tiles at a time: contexts of that size launch the one-CTA form alone."""
    h, out = Head(3, w.shape[0]), []
    for r0 in range(0, blocks * BL, h.rows):
        part = torch.zeros((h.rows, x.shape[1]), dtype=x.dtype, device=DEV)
        own = x[r0:min(r0 + h.rows, blocks * BL)]
        part[:len(own)] = own
        a, c, status, action, _ = h.run(part, w, len(own) // BL)
        assert status == 0
        out.append((a[:len(own)], c[:len(own)], action[:len(own)]))
    return [torch.cat(t) for t in zip(*out)]


def draw(hidden, vocab, rows, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    w = torch.randn((vocab, hidden), device=DEV, dtype=torch.bfloat16, generator=g).mul_(hidden ** -0.5)
    x = torch.randn((rows, hidden), device=DEV, dtype=torch.bfloat16, generator=g)
    x[::2] += 4 * w[torch.randint(0, vocab - 2, (rows // 2,), device=DEV, generator=g)]     # (half of the rows with a winner)
    return x, w


# live blocks (row tiles, form): 8 (2, pairs), 13 (4, pairs, ragged), 20 (5, one CTA a tile), 49 (13, pairs, half of the last one idle,
# ragged; hidden 768: one CTA a tile), 64 (16, pairs)
@pytest.mark.parametrize("hidden", [768, 1088, 2048])
def test_pairs_give_the_one_cta_forms_bits(hidden):
    x, w = draw(hidden, V, REQUESTS * WMAX * BL, hidden)
    h = Head(REQUESTS, V)
    for blocks in (8, 13, 20, 49, 64):
        rows = blocks * BL
        a, c, status, action, _ = h.run(x, w, blocks)
        a1, c1, action1 = one_cta(x, w, blocks)
        assert status == 0 and bool((a[rows:] == -1).all()) and not bool(c[rows:].any())
        assert torch.equal(a[:rows], a1) and torch.equal(c[:rows], c1) and torch.equal(action[:rows], action1), blocks


# rows of W that are NaN: single ones, in either half of a pair's slice, a whole slice, the last columns; behind -inf
@pytest.mark.parametrize("first,last,minus_inf", [(0, 1, 0), (127, 129, 0), (200, 201, 0), (256, 512, 0), (V - 8, V, 0), (160, 161, 160)])
def test_pairs_report_nan(first, last, minus_inf):
    x, w = draw(HIDDEN, V, REQUESTS * WMAX * BL, 3)
    x = x.abs() + 0.5                       # (a weight of -inf gives a logit of -inf)
    w[:minus_inf] = -float("inf")
    w[first:last] = float("nan")
    a, c, status, action, st = Head(REQUESTS, V).run(x, w, 64)
    assert status & B.FB_ST_NAN_LOGIT
    assert float(c.abs().max()) == 0.0 and int(action.max()) == 0 and bool((st.tokens == V - 1).all())


def test_pairs_certain_rows():
    """One logit far above the rest, up to where nothing else shows in 32 bits: every row revealed, its confidence within
    4e-6 of 1 / (1 + (V - 1) e^-d) (at most 60 additions of 2^-24 behind the term 1)."""
    rows, top = REQUESTS * WMAX * BL, V // 2 + 200
    d = torch.tensor([20.0, 26.5, 30.0, 38.0, 43.0, 50.0, 71.0, 1000.0], dtype=torch.float64)
    x, w = torch.zeros(rows, HIDDEN, dtype=torch.bfloat16), torch.zeros(V, HIDDEN, dtype=torch.bfloat16)
    x[:, 0], x[:, 1] = 1.0, d.to(torch.bfloat16).repeat(rows // 8)
    w[:, 0], w[top, 1] = -10.0, 1.0
    a, c, status, action, st = Head(REQUESTS, V).run(x.to(DEV), w.to(DEV), 64)
    want = (1 / (1 + (V - 1) * torch.exp(-d))).repeat(rows // 8)
    assert status == 0 and bool((a == top).all()) and bool((action == O.ACT_M2T).all())
    assert float((c.cpu().double() - want).abs().max()) <= 4e-6 and float(c.max()) <= 1.0


def test_pairs_give_up_report_and_recover():
    """Every wait gives up at once (no spinning), as in test_gpu_giveup.py: the launch ends by itself, says so, and the
    same context computes the same bits as before afterwards."""
    x, w = draw(HIDDEN, V, REQUESTS * WMAX * BL, 4)
    h = Head(REQUESTS, V)
    h.ctx.set_tuning(wait_cycles=-1)
    for blocks in (8, 64):
        assert h.run(x, w, blocks)[2] & B.FB_ST_DEV_TIMEOUT
    h.ctx.set_tuning()
    for blocks in (8, 64):
        a, c, status, action, _ = h.run(x, w, blocks)
        a1, c1, action1 = one_cta(x, w, blocks)
        rows = blocks * BL
        assert status == 0 and torch.equal(a[:rows], a1) and torch.equal(c[:rows], c1) and torch.equal(action[:rows], action1)


def test_form_follows_the_live_rows_under_a_graph():
    """One captured pack and head call, replayed while the live rows change: either form, the same bits as direct calls."""
    x, w = draw(1088, V, REQUESTS * WMAX * BL, 6)
    h = Head(REQUESTS, V)
    direct = {blocks: h.run(x, w, blocks) for blocks in (8, 20, 49, 4)}
    st = B.DeviceState.from_numpy(DEV, np.ones(REQUESTS, np.int32), *(np.zeros(REQUESTS, np.int32) for _ in range(3)),
                                  np.full((REQUESTS, 8 * BL), V - 1, np.int32), np.zeros((REQUESTS, WMAX), np.uint8),
                                  np.zeros((REQUESTS, 4), np.int32))
    pk, sb = B.PackBuffers.alloc(h.ctx, DEV), B.StepBuffers(h.ctx, DEV)

    def step(stream):
        B.fb_pack_wavefronts(h.ctx, st, pk, sb.ws, sb.status, stream)
        B.fb_lm_head_t2t(h.ctx, pk, x, w, st, sb.argmax, sb.conf, sb.action, sb.slot_stats, h.ws, sb.status, stream)

    side = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=side):
        step(side.cuda_stream)
    for blocks, (a, c, _, action, _) in direct.items():
        live = np.array([min(WMAX, max(0, blocks - WMAX * r)) for r in range(REQUESTS)], np.int32)
        st.R.copy_(torch.from_numpy(live))
        st.tokens.fill_(V - 1)
        graph.replay()
        torch.cuda.synchronize()
        assert int(sb.status.item()) == 0 and torch.equal(sb.argmax, a) and torch.equal(sb.conf, c) and torch.equal(sb.action, action)
