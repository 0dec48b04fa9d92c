"""The row pass at every launch shape its rule can choose: threads and CTAs per row follow the
slot capacity and the vocabulary, whose sizes here end inside a batch of loads, inside a piece
of a cluster's CTA, or below one piece per thread.  Winners bit-exact, confidence within the
parity tests' tolerance."""
import numpy as np
import pytest
import torch

from oracle import flowblock_oracle as O
from paper_2607_17652_b200 import binding as B
from paper_2607_17652_b200 import synth
from tests import harness as H
from tests import test_gpu_parity as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_requests,vocab", [
    (1, 8), (1, 1000), (1, 4096), (1, 4104), (1, 16384), (1, 16392), (1, 32768), (1, 65536), (1, 65544), (1, 151552),
    (3, 8200), (3, 40000), (11, 8200), (11, 20008), (22, 5000), (22, 8200), (70, 1032), (70, 4104),
    (22, 12008), (70, 11208), (70, 27008)])
def test_every_row_shape(n_requests, vocab):
    wl = synth.tiny_workload(n_requests=n_requests, wmax=1 if n_requests == 1 else 3, w_lo=1,
                             w_hi=1 if n_requests == 1 else 3, prefix_lo=5, prefix_hi=60, vocab=vocab)
    case = P.make_case(wl, logits_kind="normal2", with_attn=False)
    stc, z = case["stc"], case["logits"]
    rows = z.shape[0]
    rg = torch.Generator().manual_seed(vocab)
    # ties across pieces, threads and CTAs: the lowest index has to win
    top = float(z.float().max()) + 1.0
    for r in range(0, rows, 3):
        z[r, torch.randint(0, vocab, (3,), generator=rg)] = top
    ctx, st, pk, sb = P.gpu_objects(case)
    B.fb_pack_wavefronts(ctx, st, pk, sb.ws, sb.status)
    B.fb_t2t_step(ctx, pk, z.to(P.DEV), st, sb.argmax, sb.conf, sb.action, sb.slot_stats, sb.status)
    torch.cuda.synchronize()
    assert int(sb.status.item()) == 0
    opk = O.pack_wavefronts(H.oracle_cfg(stc), H.oracle_state(stc, case["tokens"]))
    xhat, conf = O.t2t_rows(H.oracle_cfg(stc), opk, H.f64(z))
    np.testing.assert_array_equal(sb.argmax.cpu().numpy(), xhat)
    assert float(np.abs(sb.conf.cpu().numpy() - conf).max()) <= P.CONF_TOL


@pytest.mark.parametrize("n_requests,vocab", [(1, 8), (1, 1000), (1, 16384), (1, 65544), (11, 20008), (70, 4104), (70, 1032)])
def test_nan_is_reported_wherever_it_stands(n_requests, vocab):
    """Rows with a NaN that no finite logit of its thread precedes: whole pieces, the head of the row, all of it
    but one logit, or behind -inf.  Each reports and reveals nothing; the rows between them are as without."""
    wl = synth.tiny_workload(n_requests=n_requests, wmax=1 if n_requests == 1 else 3, w_lo=1,
                             w_hi=1 if n_requests == 1 else 3, prefix_lo=5, prefix_hi=60, vocab=vocab)
    case = P.make_case(wl, logits_kind="normal2", with_attn=False)
    stc, z = case["stc"], case["logits"]
    opk = O.pack_wavefronts(H.oracle_cfg(stc), H.oracle_state(stc, case["tokens"]))
    live = opk.n_live * wl.block_len
    _, conf = O.t2t_rows(H.oracle_cfg(stc), opk, H.f64(z))
    nan, bad = float("nan"), list(range(0, live, 5))
    for k, r in enumerate(bad):
        if k % 5 == 0:
            z[r, :8] = nan
        elif k % 5 == 1:
            z[r, :min(vocab, 4096)] = nan
        elif k % 5 == 2:
            z[r, :vocab - 1] = nan
        elif k % 5 == 3:
            z[r, :min(vocab, 4096) - 1], z[r, min(vocab, 4096) - 1] = -float("inf"), nan
        else:
            z[r, vocab // 2:] = nan
    for rows in (bad, bad[:1], bad[1:2], bad[2:3], bad[3:4], bad[4:5]):       # together, then each kind by itself
        zz = z.clone()
        drop = [r for r in bad if r not in rows]
        zz[drop] = 0.0
        ctx, st, pk, sb = P.gpu_objects(case)
        B.fb_pack_wavefronts(ctx, st, pk, sb.ws, sb.status)
        B.fb_t2t_step(ctx, pk, zz.to(P.DEV), st, sb.argmax, sb.conf, sb.action, sb.slot_stats, sb.status)
        torch.cuda.synchronize()
        assert int(sb.status.item()) == B.FB_ST_NAN_LOGIT
        got = sb.conf.cpu().numpy()
        assert (got[rows] == 0.0).all() and int(sb.action[rows].max()) == 0
        keep = [r for r in range(live) if r not in bad]
        assert float(np.abs(got[keep] - conf[keep]).max()) <= P.CONF_TOL


@pytest.mark.parametrize("n_requests,vocab", [(1, 8), (1, 1000), (1, 65544), (11, 20008), (70, 1032), (70, 4104)])
def test_certain_rows(n_requests, vocab):
    """One logit far above the rest, up to where nothing else shows in 32 bits: never reported as NaN, revealed,
    and its confidence that of the oracle to 2e-6 (a chain of at most 32 additions behind the term 1, 2^-24 each;
    the tail's 1.4e-4 have relative errors of 1e-6)."""
    wl = synth.tiny_workload(n_requests=n_requests, wmax=1 if n_requests == 1 else 3, w_lo=1,
                             w_hi=1 if n_requests == 1 else 3, prefix_lo=5, prefix_hi=60, vocab=vocab)
    case = P.make_case(wl, logits_kind="normal2", with_attn=False)
    stc, z = case["stc"], case["logits"]
    opk = O.pack_wavefronts(H.oracle_cfg(stc), H.oracle_state(stc, case["tokens"]))
    live = opk.n_live * wl.block_len
    rg = np.random.default_rng(vocab)
    z[:] = -10.0
    for r in range(live):
        z[r, int(rg.integers(0, vocab))] = (10.0, 16.5, 20.0, 28.0, 33.0, 40.0, 61.0, 1000.0)[r % 8]
    ctx, st, pk, sb = P.gpu_objects(case)
    B.fb_pack_wavefronts(ctx, st, pk, sb.ws, sb.status)
    B.fb_t2t_step(ctx, pk, z.to(P.DEV), st, sb.argmax, sb.conf, sb.action, sb.slot_stats, sb.status)
    torch.cuda.synchronize()
    assert int(sb.status.item()) == 0
    xhat, conf = O.t2t_rows(H.oracle_cfg(stc), opk, H.f64(z))
    np.testing.assert_array_equal(sb.argmax.cpu().numpy(), xhat)
    got = sb.conf.cpu().numpy()
    assert float(np.abs(got - conf).max()) <= 2e-6 and float(got.max()) <= 1.0
    masked = opk.qtok[:live] == stc.mask_id
    assert (sb.action.cpu().numpy()[:live][masked] == O.ACT_M2T).all() and masked.any()
