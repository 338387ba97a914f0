"""The one-launch gate's scores do not depend on how many CTAs share a unit: a sequence's are the same bits alone and in a
batch of any size."""
import numpy as np
import pytest
import torch

from paper_2506_08889_b200 import binding, synth
from test_gpu_step_selection import DEV, THETA

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("g,T,dg", [(1, 1, 128), (3, 1, 64), (5, 1, 128), (8, 1, 256), (8, 1, 128), (2, 4, 128), (8, 8, 64)])
def test_scores_are_the_same_in_every_batch(g, T, dg):
    Hkv, d, b, n = 2, 128, 64, 700
    L, seed = n * b - 3, 1500 + g + T
    wq = synth.normal_bf16((Hkv, dg, g * d), seed, "wq", DEV, std=0.02)
    qn = synth.normal_bf16((140, T, Hkv * g, d), seed, "qn", DEV)
    kc = synth.normal_bf16((140, Hkv, n, dg), seed, "kc", DEV)
    ctx = binding.Context(0)
    first = []
    for B in (1, 2, 4, 9, 18, 36, 74, 140):          # clusters of sixteen CTAs down to one
        lens_t = torch.full((B,), L, dtype=torch.int32, device=DEV)
        idx = torch.zeros((B, Hkv, 9), dtype=torch.int32, device=DEV)
        cnt = torch.zeros((B, Hkv), dtype=torch.int32, device=DEV)
        sc = torch.zeros((B, Hkv, n), dtype=torch.float32, device=DEV)
        shape, gate = binding.make_shape(B, Hkv * g, Hkv, d, b, 0.09), binding.make_gate(dg, THETA, wq, None, kc[:B], n)
        before = ctx.launch_count()
        ctx.seer_gate_select_multi(shape, gate, lens_t, qn[:B], None, T, 9 * b, idx, cnt, 9, scores_out=sc)
        assert ctx.launch_count() - before == 1
        first.append(sc[0, :, :n - 1 - (T > 1)].cpu().numpy().view(np.uint32))
    for other in first[1:]:
        assert np.array_equal(first[0], other)
    assert ctx.device_status() == binding.SEER_OK

