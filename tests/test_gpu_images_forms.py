"""GPU: attention through the scratch's operand images (qwm_attend_ws without a
log-sum-exp) at full sizes and in every form its work is shared out: whole
waves of query blocks, a tail in equal parts per block, a tail flattened over
the CTAs, and more heads than one scratch of images holds.

The form is taken from the rule restated here and asserted where the GPU has
the SM count it was computed for.  Sampled rows of sampled heads are compared
with the oracle's fp64 softmax (2e-2 at most, 2e-3 on average); every output
with the kernel that rebuilds its keys itself: 2e-2, and a bf16 ulp of each
rounding (2^-7 relative).
"""
import math

import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2609_26425_gb300 import synth
import paper_2609_26425_gb300 as qwm

from parity import compare_attention, oracle_append, oracle_kv, strided_centroids
from test_gpu_fullsize import sample_rows

pytestmark = pytest.mark.gpu


def tail_form(Nq, heads, Nk, nsm):
    """(whole waves, form of the tail, does the flattened tail leave a remainder)."""
    NT, units = -(-Nk // 128), heads * -(-Nq // 256)
    waves, n = units // nsm, units % nsm
    if n == 0:
        return waves, "none", False
    T = n * NT
    s = nsm // n
    per = max(-(-NT // s), 3)
    s = -(-NT // per)
    g = min(max(-(-T // 3), n), nsm)
    if per + (12 if s > 1 else 4) <= -(-T // g) + 24:
        return waves, "parts" if s > 1 else "whole", False
    return waves, "flat", T % g != 0


def image_heads(H, Nk):
    """Heads whose images are in the scratch together."""
    most = (2 << 30) // (-(-Nk // 128) * 65536)
    n = -(-H // most)
    return -(-H // n)


@pytest.mark.parametrize("H,chunks,C,r,Nq,Ncur,heads,form", [
    (40, [4680] * 6, 256, 16, 4680, 4680, (0, 23, 39), (5, "none", False)),       # the Wan-14B layer
    (12, [880] * 15, 64, 32, 880, 880, (0, 11), (0, "parts", False)),             # the 15-chunk window
    (80, [3200, 3200], 4, 16, 200, 0, (0, 1, 40, 79), (0, "flat", True)),         # CTAs run across blocks
    (80, [4000, 3296], 4, 8, 250, 0, (0, 39, 79), (0, "flat", False)),            # the same, equal shares
    (58, [3200, 3200], 4, 16, 1000, 0, (0, 37, 38, 57), (1, "flat", True)),       # after a whole wave
    (81, [20000], 4, 8, 300, 33700, (0, 40, 41, 80), (0, "flat", True)),          # two groups: 41 and 40 heads
    (40, [4680] * 14, 256, 16, 1024, 1024, (0, 18, 39), (1, "parts", False)),     # a long history
    (4, [880] * 15, 64, 16, 128, 0, (0, 3), (0, "parts", False)),                 # 35 parts of a block
    (1, [1000] * 40, 16, 8, 130, 0, (0,), (0, "parts", False)),                   # 105 parts
    (6, [300, 900], 16, 16, 250, 0, (0, 5), (0, "parts", False)),                 # 4 parts
])
def test_images_forms_match_oracle_and_plain(H, chunks, C, r, Nq, Ncur, heads, form):
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    Nk = sum(chunks) + Ncur
    per_group = image_heads(H, Nk)
    assert (per_group < H) == (H == 81)
    if nsm == 152:
        for n in {per_group, H - (H - 1) // per_group * per_group}:
            assert tail_form(Nq, n, Nk, nsm) == form
    heads, G, M = list(heads), 32, 4
    g = torch.Generator(device="cuda").manual_seed(H * Nq)

    def rows(n):
        return torch.randn(n, H, 128, generator=g, device="cuda")

    def keys(n):
        k = rows(n)
        k[:, :, [5, 40, 77, 120]] *= 8
        return k.bfloat16()

    cfg = qwm.config(H, C, group_size=G, psac_rank=r, candidates=M)
    cache = qwm.Cache(cfg, max(chunks), len(chunks))
    Ks, Vs = [], []
    for i, N in enumerate(chunks):
        k, v = keys(N), rows(N).bfloat16()
        idx = torch.arange(C) * N // C
        kc, vc = (x[idx.cuda()].transpose(0, 1).contiguous() for x in (k, v))
        U = synth.random_orthonormal(80 + i, H, 128, r).contiguous()
        qwm.qwm_quantize_append(cfg, cache, k, v, kc, vc, U=U.cuda())
        kb, vb = (synth.bits(x[:, heads].cpu().contiguous()) for x in (k, v))
        Ub = np.ascontiguousarray(synth.bits(U)[heads])
        kcb, vcb = strided_centroids(kb, C), strided_centroids(vb, C)
        ko, vo = oracle_append(kb, vb, kcb, vcb, G=G, r=r, M=M, U_bits=Ub)
        K, V = oracle_kv(ko, vo, kcb, vcb, G=G, r=r, U_bits=Ub)
        Ks.append(K)
        Vs.append(V)
    q = rows(Nq).bfloat16()
    kd, vd = (keys(Ncur), rows(Ncur).bfloat16()) if Ncur else (None, None)
    if Ncur:
        Ks.append(orc.bf16_to_f32(synth.bits(kd[:, heads].cpu().contiguous())).astype(np.float64))
        Vs.append(orc.bf16_to_f32(synth.bits(vd[:, heads].cpu().contiguous())).astype(np.float64))
    ws = qwm.attend_workspace(cfg, cache, Nq, Ncur)
    assert ws.numel() >= per_group * -(-Nk // 128) * 65536   # the images' path runs
    out = qwm.qwm_attend(cfg, cache, q, kd, vd, workspace=ws)
    plain = qwm.qwm_attend(cfg, cache, q, kd, vd)
    torch.cuda.synchronize()
    assert cache.status() == 0
    at = sample_rows(Nq, 24, H)
    ref, _ = orc.attend(synth.bits(q[:, heads].cpu().contiguous()), np.concatenate(Ks), np.concatenate(Vs),
                        1 / math.sqrt(128), rows=at)
    compare_attention(out.float().cpu().numpy()[at][:, heads], ref)
    a, b = out.float(), plain.float()
    assert ((a - b).abs() <= 2e-2 + 2.0 ** -6 * b.abs()).all()
