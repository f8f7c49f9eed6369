"""GPU: attention through the scratch buffer's operand images (qwm_attend_ws
without a log-sum-exp) against the oracle and against the kernel without
scratch, at the sizes where the images' packing, the query blocks and the
split of the key tiles can go wrong."""
import pytest
import torch

import paper_2609_26425_gb300 as qwm
from paper_2609_26425_gb300 import synth
from parity import compare_attention
from test_gpu_parity import build_cache_and_reference, dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,chunks,C,G,r,Ncur,Nq,sf", [
    (1, [500, 13], 4, 32, 16, 0, 1, 0),              # one query; keys end on a tile boundary + 1
    (2, [127, 1, 384], 16, 32, 8, 0, 128, 0),        # the fewest keys; one whole Q tile
    (2, [256, 256], 16, 64, 32, 128, 129, 0),        # whole tiles only; one query in the second Q tile
    (3, [300, 277, 5], 16, 64, 16, 130, 257, 1),     # ragged chunks, a block with a single query
    (5, [200, 333], 64, 32, 0, 257, 700, 0),         # no PSAC
    (2, [640, 640, 640], 100, 32, 32, 0, 300, 1),    # two-level scales, split tiles
    (70, [400, 240], 4, 32, 8, 0, 520, 0),           # more query blocks than SMs: whole waves and a tail
    (80, [400, 900], 4, 32, 16, 0, 300, 0),          # a tail whose CTAs run across blocks
    (2, [1024], 4, 32, 16, 0, 40, 0),                # a single chunk
])
def test_images_attend_matches_oracle_and_plain(H, chunks, C, G, r, Ncur, Nq, sf):
    """Within the attention tolerance of the oracle's fp64 softmax (2e-2 at
    most, 2e-3 on average), and of the kernel without scratch; twice the same bits."""
    rows = None if H * Nq < 10000 else list(range(0, Nq, 37))
    cfg, cache, q, kc, vc, ref, _ = build_cache_and_reference(H, chunks, C, G, r, 4, seed=11 * H + Nq, Ncur=Ncur, Nq=Nq,
                                                             scale_format=sf, rows=rows)
    kd, vd = (dev(kc), dev(vc)) if Ncur else (None, None)
    ws = qwm.attend_workspace(cfg, cache, Nq, Ncur)
    out = qwm.qwm_attend(cfg, cache, dev(q), kd, vd, workspace=ws)
    plain = qwm.qwm_attend(cfg, cache, dev(q), kd, vd)
    ws.fill_(0x7F)                                   # nothing is kept in the scratch between calls
    again = qwm.qwm_attend(cfg, cache, dev(q), kd, vd, workspace=ws)
    torch.cuda.synchronize()
    assert cache.status() == 0
    assert torch.equal(out, again)
    got = out.float().cpu().numpy()
    compare_attention(got if rows is None else got[rows], ref)
    assert (out.float() - plain.float()).abs().max().item() < 2e-2


def test_images_attend_reports_values_beyond_binary16():
    """A Query, an active Key and an active Value beyond binary16 are each
    reported (QWM_ERR_NONFINITE) and saturate: the output stays finite."""
    cfg, cache, q, kc, vc, _, _ = build_cache_and_reference(2, [500], 16, 32, 16, 4, seed=3, Ncur=100, Nq=60)
    ws = qwm.attend_workspace(cfg, cache, 60, 100)
    for which in range(3):
        x = [q.clone(), kc.clone(), vc.clone()]
        x[which][7, 1, 3] = 1.0e5
        out = qwm.qwm_attend(cfg, cache, *(dev(t) for t in x), workspace=ws)
        torch.cuda.synchronize()
        assert cache.status() == 6
        assert torch.isfinite(out.float()).all()
    qwm.qwm_attend(cfg, cache, dev(q), dev(kc), dev(vc), workspace=ws)
    assert cache.status() == 0
