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
