"""Key tiles of the attention at their edges: ragged tiles (taken 32 columns at
a time) next to full ones (taken whole), and full tiles of 8-bit pages that
break the bound on their exponentials and are taken again.  Tolerances are
those of the parity tests the helpers come from."""
import numpy as np
import pytest
import torch

from paper_2607_17652_b200 import synth
from tests import harness as H
from tests import test_gpu_fp8 as F
from tests import test_gpu_parity as P

pytestmark = pytest.mark.gpu
EDGES = (1, 31, 32, 33, 63, 64, 96, 97, 127, 128, 129, 256)


def _workload(prefix, **kw):
    w = 1 + prefix % 3
    return synth.tiny_workload(n_requests=2, wmax=3, w_lo=w, w_hi=w, prefix_lo=prefix, prefix_hi=prefix, **kw)


@pytest.mark.parametrize("prefix", EDGES)
@pytest.mark.parametrize("head_dim", [64, 128])
def test_ragged_and_full_tiles(prefix, head_dim):
    P.run_attention(P.make_case(_workload(prefix, head_dim=head_dim), with_logits=False))


@pytest.mark.parametrize("prefix", EDGES)
def test_ragged_and_full_tiles_of_8_bit_pages(prefix):
    c = F._setup(_workload(prefix, head_dim=128))
    out, ref, rows = F._run(c)
    rel, worst = F._within_f8_bound(c, out, ref, rows)
    assert rel <= F.F8_REL_L2 and worst <= 1.0, (rel, worst)


@pytest.mark.parametrize("where", [7, 140, 255, 300])
def test_8_bit_reference_moves_to_a_dominant_key(where):
    """All queries point along one +-1 direction and one key holds a multiple of it, so that key's
    weight is 1 and both 8-bit roundings are exact whichever tile (first, full, ragged last)
    makes the reference move: what is left is the rounding of the output."""
    wl = synth.tiny_workload(n_requests=3, wmax=3, w_lo=1, w_hi=3, prefix_lo=330, prefix_hi=380, head_dim=128)
    c = F._setup(wl)
    rng = np.random.default_rng(3)
    direction = torch.from_numpy(rng.choice([-1.0, 1.0], size=128)).to(torch.float32)
    big = (direction * 448.0).to(torch.float8_e4m3fn).view(torch.uint8)
    k8 = c["k8"].clone()
    for r in range(wl.n_requests):
        k8[int(c["stc"].page_table[r, where // 64]), :, where % 64, :] = big
    q = (direction * 0.5).to(torch.bfloat16).expand_as(c["q"]).contiguous()
    out, ref, rows = F._run(c, q=q, k8=k8, scatter=False)
    max_abs, rel = H.attn_errors(out, ref, rows)
    # half a bf16 ulp of the largest output is 2^-9 of it; twice that for the fp32 normalisation
    assert max_abs <= 2 ** -8 * float(np.abs(ref[rows]).max()) and rel <= 5e-3, (max_abs, rel)
