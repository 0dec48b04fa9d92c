"""The split of the key axis that is chosen by estimate: the device builds the list that the host
mirror of the arithmetic announces, whatever the batch (few or many units, short or long, with
leftover tiles, more requests than one pass of the scheduler block), and the attention over
it agrees with the unsplit one."""
import numpy as np
import pytest
import torch

from paper_2607_17652_b200 import binding as B
from paper_2607_17652_b200 import synth

DEV = "cuda:0"


def _cfg(**over):
    return dict(dict(max_requests=64, wmax=4, block_len=32, n_q_heads=32, n_kv_heads=8, head_dim=128, page_size=64,
                     num_pages=64 * 520, max_pages_per_req=520, vocab=1024, mask_id=1023, eos_id=1022, max_blocks=32,
                     s_pe=1, tau_mask=0.9, tau_edit=0.95, theta_spawn=0.5, sm_scale=0.0), **over)


def test_estimated_split_fits_and_leaves_nothing_out():
    rg = np.random.default_rng(11)
    ctx = B.Context(**_cfg())
    for _ in range(400):
        n = int(rg.integers(1, 65))
        P = rg.integers(0, int(2 ** rg.uniform(5, 15)), size=n)
        w = rg.integers(0, 5, size=n)
        pl = ctx.attn_plan(P, w)
        assert pl["parts"] <= pl["max_parts"] and pl["units"] <= pl["max_units"] and pl["items"] <= pl["max_items"], pl
        assert pl["items"] >= pl["units"]
    # 160 long units for 148 SMs: the second wave would run nearly empty, pieces fill it
    assert ctx.attn_plan([16000] * 10, [4] * 10)["parts"] > 0
    # three full waves of short items: nothing to gain
    assert ctx.attn_plan([300] * 28, [4] * 28)["parts"] == 0


def test_eight_bit_pages_are_not_split_by_estimate():
    # (their weights are rounded against a reference per piece: another split, another rounding)
    rg = np.random.default_rng(12)
    fp8 = dict(kv_fp8=1, window_in_pages=1)
    ctx, fixed = B.Context(**_cfg(**fp8)), B.Context(tuning=dict(attn_target_items=296, attn_min_chunk_tiles=4), **_cfg(**fp8))
    for _ in range(100):
        n = int(rg.integers(1, 65))
        P, w = rg.integers(0, int(2 ** rg.uniform(5, 15)), size=n), rg.integers(0, 5, size=n)
        assert ctx.attn_plan(P, w) == fixed.attn_plan(P, w)


def test_short_contexts_have_no_pieces():
    # rows of 10 and 11 pages: a prefix of 608 / 672 tokens and a window of one block, 6 / 7 key tiles
    plan = lambda tuning, pages: B.Context(tuning=tuning, **_cfg(max_pages_per_req=pages)).attn_plan([128] * 2, [4] * 2)
    assert plan(None, 10)["max_parts"] == 0 and plan(None, 10)["parts"] == 0
    assert plan(None, 11)["max_parts"] > 0
    # what the caller asks for is done
    assert plan(dict(attn_target_items=8), 10)["max_parts"] > 0
    assert plan(dict(attn_min_chunk_tiles=1), 10)["max_parts"] > 0


def _tiles(P, w):           # key tiles of a request's units (window beside the pages, one Q tile per slot)
    return -(-P // 128) + -(-(w * 32) // 128)


@pytest.mark.parametrize("min_chunk", [1, 3, 8, 62, 64, 128, 300, 1000])
def test_callers_shortest_range_holds_without_a_target(min_chunk):
    # batches large enough for filler pieces at the end of the list
    rg = np.random.default_rng(min_chunk)
    for pages in (124, 260, 520):
        ctx = B.Context(tuning=dict(attn_min_chunk_tiles=min_chunk), **_cfg(max_pages_per_req=pages))
        for _ in range(40):
            n = int(rg.integers(19, 65))
            lo = int(rg.integers(0, pages * 64 - 128))
            P = rg.integers(lo, pages * 64 - 127, size=n)
            pl = ctx.attn_plan(P, [4] * n)
            assert pl["parts"] <= pl["max_parts"] and pl["items"] <= pl["max_items"], (pl, P)
            # 16 units a request, cut into no more than ceil(tiles / shortest) pieces each
            pieces = sum(16 * -(-_tiles(int(x), 4) // min_chunk) for x in P)
            assert pl["items"] <= pieces, (pl, P)
            if min_chunk >= _tiles(int(P.max()), 4):
                assert pl["parts"] == 0 and pl["items"] == 16 * n, (pl, P)


@pytest.mark.gpu
@pytest.mark.parametrize("seed", [36154492, 54453613, 40045238, 42664750, 51996146, 31555111, 63399331])
def test_near_ties_of_the_estimate(seed):
    # batches in which the two best chunk lengths are estimated within a unit in the last place of each other:
    # device and host have to round alike to agree on one
    def draw():
        nonlocal seed
        seed = (seed * 1664525 + 1013904223) & 0xFFFFFFFF
        return seed >> 8
    n, hi = 60 + draw() % 40, 3000 + draw() % 6000
    P, w = zip(*[(draw() % hi, 1 + draw() % 4) for _ in range(n)])
    ctx = B.Context(**_cfg(max_requests=n, n_q_heads=12, n_kv_heads=3, max_pages_per_req=150))
    st = B.DeviceState.from_numpy(DEV, np.ones(n, np.int32), np.array(P, np.int32), np.zeros(n, np.int32),
                                  np.array(w, np.int32), np.zeros((n, 32 * 32), np.int32), np.zeros((n, 4), np.uint8),
                                  np.zeros((n, 150), np.int32))
    pk, sb = B.PackBuffers.alloc(ctx, DEV), B.StepBuffers(ctx, DEV)
    B.fb_pack_wavefronts(ctx, st, pk, sb.ws, sb.status)
    torch.cuda.synchronize()
    assert int(sb.status.item()) == 0
    hdr, plan = sb.ws[:64].cpu().numpy().view(np.int32), ctx.attn_plan(P, w)
    assert (int(hdr[1]), int(hdr[0]), int(hdr[3])) == (plan["units"], plan["items"], plan["parts"])


@pytest.mark.gpu
@pytest.mark.parametrize("min_chunk", [0, 8, 30, 64])
def test_shortest_range_on_the_device(min_chunk):
    # 300 units of 34 to 45 key tiles; with 64 no range may be cut and the context has no room for pieces
    wl = synth.tiny_workload(n_requests=50, wmax=4, w_lo=4, w_hi=4, prefix_lo=4200, prefix_hi=5600, head_dim=64,
                             n_q_heads=12, n_kv_heads=3)
    _plan_and_attention(wl, (dict(attn_min_chunk_tiles=min_chunk), dict(attn_target_items=1)), 0)


@pytest.mark.gpu
@pytest.mark.parametrize("n_requests,prefix,w,resident", [
    (1, (64, 64), (2, 2), 0), (1, (3001, 3001), (1, 1), 1), (2, (9000, 12000), (3, 3), 0), (9, (100, 2500), (1, 4), 1),
    (20, (1500, 4000), (1, 3), 0), (60, (100, 900), (1, 4), 0), (1100, (1, 200), (1, 1), 0)])
def test_device_builds_the_announced_list(n_requests, prefix, w, resident):
    wl = synth.tiny_workload(n_requests=n_requests, wmax=4, w_lo=w[0], w_hi=w[1], prefix_lo=prefix[0],
                             prefix_hi=prefix[1], head_dim=128, n_q_heads=12, n_kv_heads=3)
    _plan_and_attention(wl, (None, dict(attn_target_items=1)), resident)


def _plan_and_attention(wl, tunings, resident):
    stc = synth.make_structure(wl)
    tokens = synth.make_tokens(stc)
    q, kw, vw, kp, vp = (t.to(DEV) for t in synth.make_attn_inputs(stc))
    if resident:
        kw = vw = None
    outs = []
    for tuning in tunings:
        ctx = B.Context(tuning=tuning, **synth.config_dict(stc, window_in_pages=resident))
        st = B.DeviceState.from_numpy(DEV, stc.active, stc.prefix_len, stc.L, stc.R, tokens,
                                      np.zeros((wl.n_requests, wl.wmax), np.uint8), stc.page_table)
        pk = B.PackBuffers.alloc(ctx, DEV)
        sb = B.StepBuffers(ctx, DEV)
        B.fb_pack_wavefronts(ctx, st, pk, sb.ws, sb.status)
        for _ in range(2):                        # the work ticket is re-armed by the launch itself
            sb.out.fill_(7.0)
            B.fb_wavefront_attn(ctx, pk, q, kw, vw, kp, vp, st.page_table, sb.out, sb.ws, sb.status)
        torch.cuda.synchronize()
        assert int(sb.status.item()) == 0
        hdr = sb.ws[:64].cpu().numpy().view(np.int32)          # n_items, n_units, chunk length, n_parts
        plan = ctx.attn_plan(stc.prefix_len, stc.R - stc.L)
        assert (int(hdr[1]), int(hdr[0]), int(hdr[3])) == (plan["units"], plan["items"], plan["parts"])
        outs.append(sb.out.float())
    # two schedules of the same sums: the weights are rounded to bf16 against different references
    # (2^-9 each) and the output once more
    err = float((outs[0] - outs[1]).norm() / outs[1].norm())
    assert err <= 4 * 2 ** -9, err


@pytest.mark.gpu
@pytest.mark.parametrize("n_requests,w,kv_heads,prefix", [
    (1, 2, 8, 3001), (1, 3, 8, 28123), (8, 2, 4, 900), (9, 2, 4, 900), (37, 1, 4, 700), (37, 2, 4, 700), (38, 1, 8, 700),
    (31, 3, 3, 2500), (33, 3, 3, 2500), (600, 1, 1, 300)])
def test_list_holds_every_key_range_once(n_requests, w, kv_heads, prefix):
    # one request (not sorted), few requests and many, 148 items and more, odd KV heads
    tiles_per_slot, wmax, blocks = 1, 3, 8
    ctx = B.Context(**_cfg(max_requests=n_requests, wmax=wmax, n_q_heads=4 * kv_heads, n_kv_heads=kv_heads, max_blocks=blocks,
                           max_pages_per_req=450))
    P = np.maximum(prefix - 64 * np.arange(n_requests), prefix // 2).astype(np.int32)
    st = B.DeviceState.from_numpy(DEV, np.ones(n_requests, np.int32), P, np.zeros(n_requests, np.int32),
                                  np.full(n_requests, w, np.int32), np.zeros((n_requests, blocks * 32), np.int32),
                                  np.zeros((n_requests, wmax), np.uint8), np.zeros((n_requests, 450), np.int32))
    pk, sb = B.PackBuffers.alloc(ctx, DEV), B.StepBuffers(ctx, DEV)
    B.fb_pack_wavefronts(ctx, st, pk, sb.ws, sb.status)
    torch.cuda.synchronize()
    assert int(sb.status.item()) == 0
    plan, ws = ctx.attn_plan(P, np.full(n_requests, w)), sb.ws.cpu().numpy()
    n_items, n_units, _, n_parts, _, ticket, done, most = ws[:32].view(np.int32)
    assert (n_units, n_items, n_parts) == (plan["units"], plan["items"], plan["parts"]) and ticket == done == 0
    at = 256 + -(-plan["max_items"] * 32 // 256) * 256
    items = ws[256:256 + 32 * n_items].view(np.int32).reshape(-1, 8)
    units = ws[at:at + 64 * n_units].view(np.int32).reshape(-1, 16)
    chunks, n_tiles, part_base = units[:, 7], units[:, 6], units[:, 10]
    assert most == chunks.max() and (units[items[:, 0], 0] == items[:, 4]).all()
    # every unit's key tiles once, in its pieces' order
    order = np.lexsort((items[:, 1], items[:, 0]))
    it, k = items[order], 0
    for u in range(n_units):
        own = it[k:k + chunks[u]]
        k += chunks[u]
        assert (own[:, 0] == u).all() and (own[:, 1] == np.arange(chunks[u])).all()
        assert own[0, 2] == 0 and own[-1, 3] == n_tiles[u] and (own[1:, 2] == own[:-1, 3]).all() and (own[:, 3] > own[:, 2]).all()
    assert k == n_items
    # split units have places of their own for their pieces
    assert (part_base[chunks <= 1] == -1).all()
    split = np.argsort(part_base)[(chunks <= 1).sum():]
    assert (part_base[split][1:] >= (part_base + chunks)[split][:-1]).all()
    # every (slot, KV head) once, as tile A or B
    tiles = [(u[2], u[1] & 0xffff, u[4]) for u in units] + [(u[3], u[1] >> 16, u[5]) for u in units if u[3] >= 0]
    assert len(set(tiles)) == len(tiles) == n_requests * w * kv_heads * tiles_per_slot
    if n_requests > 1:          # longest first
        assert (np.diff(items[:, 3] - items[:, 2]) <= 1).all()



# windows and whether a request is decoding; one request with work among many rows, few and many, odd KV heads, requests without
# units between others, blocks of one and two Q tiles, the window beside the pages and in them
@pytest.mark.gpu
@pytest.mark.parametrize("resident", [0, 1])
@pytest.mark.parametrize("block_len,kv_heads,windows,prefix", [
    (32, 8, [0, 0, 0, 0, 0, 2, 0, 0], 3001), (64, 3, [-3, 0, 0, 1], 9000), (32, 4, [0, 3, 0, 0, -2, 0, 1, 0], 5000),
    (64, 8, [1, 0, 3, 2, 0, 0, 3, 1], 1500), (32, 1, [0] * 7 + [3], 300), (32, 3, [0] * 20 + [2], 4000),
    (64, 3, [0, 1, 2, 3, -1] * 6, 2500), (32, 5, [3, 0, 0, 1] * 150, 700), (32, 8, [0] * 8, 500), (32, 8, [0] * 9, 500)])
def test_list_of_a_mixed_batch(resident, block_len, kv_heads, windows, prefix):
    n, wmax, blocks, G = len(windows), 3, 8, 4
    ctx = B.Context(**_cfg(max_requests=n, wmax=wmax, block_len=block_len, n_q_heads=G * kv_heads, n_kv_heads=kv_heads,
                           max_blocks=blocks, max_pages_per_req=160, window_in_pages=resident))
    rg = np.random.default_rng(n * block_len + kv_heads)
    P, w = rg.integers(prefix // 3, prefix + 1, n).astype(np.int32), np.abs(windows).astype(np.int32)
    st = B.DeviceState.from_numpy(DEV, np.array([x >= 0 for x in windows], np.int32), P, np.zeros(n, np.int32), w,
                                  np.zeros((n, blocks * block_len), np.int32), np.zeros((n, wmax), np.uint8),
                                  np.zeros((n, 160), np.int32))
    w = np.maximum(windows, 0)                       # (a request that is not decoding has no window)
    pk, sb = B.PackBuffers.alloc(ctx, DEV), B.StepBuffers(ctx, DEV)
    B.fb_pack_wavefronts(ctx, st, pk, sb.ws, sb.status)
    torch.cuda.synchronize()
    assert int(sb.status.item()) == 0 and int(pk.n_live.item()) == w.sum()
    plan, ws = ctx.attn_plan(P, w), sb.ws.cpu().numpy()
    n_items, n_units, _, n_parts, total, _, _, most = ws[:32].view(np.int32)
    assert (n_units, n_items, n_parts) == (plan["units"], plan["items"], plan["parts"])
    at = 256 + -(-plan["max_items"] * 32 // 256) * 256
    items = ws[256:256 + 32 * n_items].view(np.int32).reshape(-1, 8)
    units = ws[at:at + 64 * n_units].view(np.int32).reshape(-1, 16)
    slot_req, slot_s = pk.slot_req.cpu().numpy(), pk.slot_s.cpu().numpy()
    up = lambda a, b: -(-a // b)
    tiles, per = [], block_len * G // 128
    for u, (req, kvh, slot_a, slot_b, t0_a, t0_b, n_tiles, chunks, nvis_a, nvis_b, part, pre, npt, _, win_a, win_b) in enumerate(units):
        window = w[req] * block_len
        assert w[req] > 0 and pre == P[req]
        assert n_tiles == (up(P[req] + window, 128) if resident else up(P[req], 128) + up(window, 128))
        assert npt == (n_tiles if resident else up(P[req], 128))
        for slot, t0, nvis, win, kv in ((slot_a, t0_a, nvis_a, win_a, kvh & 0xffff), (slot_b, t0_b, nvis_b, win_b, kvh >> 16)):
            if slot < 0:
                assert slot == slot_b and nvis == 0
                continue
            assert slot_req[slot] == req and win == (slot_s[slot] + 1) * block_len and t0 in range(0, block_len, 128 // G)
            assert nvis == (up(P[req] + win, 128) if resident else npt + up(win, 128))
            tiles.append((slot, t0, kv))
        own = items[items[:, 0] == u]
        own = own[np.argsort(own[:, 1])]
        edges = np.arange(chunks + 1) * n_tiles // chunks
        assert len(own) == chunks and (own[:, 2] == edges[:-1]).all() and (own[:, 3] == edges[1:]).all() and (own[:, 4] == req).all()
        assert part == -1 if chunks <= 1 else 0 <= part <= n_parts - chunks
    assert len(items) == units[:, 7].sum() and len(set(tiles)) == len(tiles) == w.sum() * kv_heads * per
    assert total == (units[:, 6]).sum() and (most == units[:, 7].max() if n_units else most == 0)
    # the most costly first, but for one request's few, which come unit by unit
    if n_units:
        nv = units[items[:, 0]][:, 8:10]
        n_ab = np.clip(np.minimum(items[:, 3:4], nv) - items[:, 2:3], 0, None)
        cost = (6 * n_ab.max(1) + n_ab.min(1) + 1) >> 1
        if n <= 8 and (w > 0).sum() == 1 and n_items <= 148:
            assert (np.diff(items[:, 0]) >= 0).all() and (items[:, 1] == np.concatenate([np.arange(c) for c in units[:, 7]])).all()
        else:
            assert (np.diff(cost) <= 0).all()


@pytest.mark.gpu
@pytest.mark.parametrize("max_requests", [1, 2, 9])
@pytest.mark.parametrize("tiles", [(1 << 19) - 2, (1 << 19) - 1, (1 << 20) + 5, 11423809, 13823826, 16777000])
def test_cuts_of_a_very_long_range(max_requests, tiles):
    # quotients on both sides of the 2^20 up to which they are taken by reciprocal, and near the largest prefix
    # (the call reads neither the pages nor the page table)
    ctx = B.Context(**_cfg(max_requests=max_requests, wmax=1, block_len=64, n_q_heads=2, n_kv_heads=1, head_dim=64, max_blocks=2,
                           max_pages_per_req=2 * tiles + 2))
    P = np.zeros(max_requests, np.int32)
    w = np.zeros(max_requests, np.int32)
    P[-1], w[-1] = 128 * tiles, 1
    st = B.DeviceState.from_numpy(DEV, np.ones(max_requests, np.int32), P, np.zeros(max_requests, np.int32), w,
                                  np.zeros((max_requests, 2 * 64), np.int32), np.zeros((max_requests, 1), np.uint8),
                                  np.zeros((max_requests, 4), np.int32))
    pk, sb = B.PackBuffers.alloc(ctx, DEV), B.StepBuffers(ctx, DEV)
    B.fb_pack_wavefronts(ctx, st, pk, sb.ws, sb.status)
    torch.cuda.synchronize()
    assert int(sb.status.item()) == 0
    plan, ws = ctx.attn_plan(P, w), sb.ws.cpu().numpy()
    n_items, n_units, _, n_parts = ws[:16].view(np.int32)
    assert (n_units, n_items, n_parts) == (plan["units"], plan["items"], plan["parts"]) and n_items > 1
    items = ws[256:256 + 32 * n_items].view(np.int32).reshape(-1, 8)
    items = items[np.argsort(items[:, 1])]
    edges = np.arange(n_items + 1, dtype=np.int64) * (tiles + 1) // n_items
    assert (items[:, 1] == np.arange(n_items)).all()
    assert (items[:, 2] == edges[:-1]).all() and (items[:, 3] == edges[1:]).all()
