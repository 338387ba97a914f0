"""The one-launch gate's compressed keys on their way through the K/V ring: tiles of 16 keys, as many slots as the scores leave
room for (fewer than there are warps, more, each used once or several times), a last tile that the cache's end cuts short."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2506_08889_b200 import binding, synth
from test_gpu_step_selection import DEV, THETA, scores64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hkv,g,T,dg,n", [
    (1, 1, 4, 1, 128, 1),              # one key
    (1, 1, 4, 1, 64, 17),              # a tile and one key of the next; CTAs without any
    (1, 2, 8, 1, 256, 121),            # the last tile ends in its second half ...
    (1, 2, 8, 3, 128, 133),            # ... and in its first
    (4, 8, 4, 1, 128, 2047),           # slots used twice
    (1, 1, 8, 1, 256, 8187),           # fewer slots than warps
    (2, 80, 2, 1, 128, 8192),          # one CTA a unit, the most keys of the gate alone: slots used 40 times
    (2, 80, 2, 1, 64, 4099),
    (2, 40, 4, 4, 256, 4100),          # several query tokens
])
def test_scores_of_every_key(B, Hkv, g, T, dg, n):
    b, d = 16, 128
    L = (n + 3) * b + 5                # the cache ends before the sequence does: all n keys are candidates
    seed = 900 + n + dg
    qn = synth.normal_bf16((B, T, Hkv * g, d), seed, "qn", DEV)
    wq = synth.normal_bf16((Hkv, dg, g * d), seed, "wq", DEV, std=0.02)
    kc = synth.normal_bf16((B, Hkv, n, dg), seed, "kc", DEV)
    sel = min(40, n + 1)
    ctx = binding.Context(0)
    lens_t = torch.full((B,), L, dtype=torch.int32, device=DEV)
    idx = torch.zeros((B, Hkv, sel), dtype=torch.int32, device=DEV)
    cnt = torch.zeros((B, Hkv), dtype=torch.int32, device=DEV)
    sc = torch.zeros((B, Hkv, n), dtype=torch.float32, device=DEV)
    shape, gate = binding.make_shape(B, Hkv * g, Hkv, d, b, 0.09), binding.make_gate(dg, THETA, wq, None, kc, n)
    before = ctx.launch_count()
    for _ in range(3):                 # (one right behind the other)
        ctx.seer_gate_select_multi(shape, gate, lens_t, qn, None, T, sel * b, idx, cnt, sel, scores_out=sc)
    assert ctx.launch_count() - before == 3
    torch.cuda.synchronize()
    assert ctx.device_status() == binding.SEER_OK
    want = scores64(qn, wq, kc, L)
    # a sum of d_gate products of the size of the scores, each rounded to 2^-24 at most a few times
    err = (sc.double() - want).abs().amax((0, 1)).cpu().numpy()
    bad = np.nonzero(err > 8 * 2.0 ** -24 * math.sqrt(dg) * float(want.abs().max()))[0]
    assert bad.size == 0, (bad[:8], err[bad[:8]])
