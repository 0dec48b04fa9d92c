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
