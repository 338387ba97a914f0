"""The one-launch gate's scores do not depend on how many CTAs share a unit: a sequence's are the same bits alone and in a
batch of any size.  And gate queries next to the largest fp32 number stay finite."""
import numpy as np
import pytest
import torch

from paper_2506_08889_b200 import binding, synth
from test_gpu_step_selection import DEV, THETA, scores64

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


def test_gate_query_next_to_the_largest_number():
    # channel 63 of 128 turns by 4800 * theta^(-126/128) = 0.006: the query's channel is 3.4e38 * cos, above the largest bf16
    g, d, dg, b, n = 1, 128, 128, 16, 300
    L = n * b - 3
    qn = torch.zeros((1, 1, g, d), dtype=torch.bfloat16, device=DEV)
    qn[..., 0], qn[..., 64] = 3.3895314e38, 1.0e36
    wq = torch.zeros((1, dg, g * d), dtype=torch.bfloat16, device=DEV)
    wq[:, 63, 0] = wq[:, 63, 64] = 1.0
    kc = torch.zeros((1, 1, n, dg), dtype=torch.bfloat16, device=DEV)
    kc[..., 63] = (torch.arange(n, device=DEV) % 37 - 18) * 2.0 ** -90
    lens_t = torch.tensor([L], dtype=torch.int32, device=DEV)
    idx, cnt = torch.zeros((1, 1, 40), dtype=torch.int32, device=DEV), torch.zeros((1, 1), dtype=torch.int32, device=DEV)
    sc = torch.zeros((1, 1, n), dtype=torch.float32, device=DEV)
    ctx = binding.Context(0)
    shape, gate = binding.make_shape(1, g, 1, d, b, 0.09), binding.make_gate(dg, THETA, wq, None, kc, n)
    before = ctx.launch_count()
    ctx.seer_gate_select(shape, gate, lens_t, qn[:, 0], None, 40 * b, idx, cnt, 40, scores_out=sc)
    assert ctx.launch_count() - before == 1
    want = scores64(qn, wq, kc, L)[0, 0, :n - 1]
    assert float(want.abs().max()) > 1e11
    assert bool(((sc[0, 0, :n - 1].double() - want).abs() <= 4 * 2.0 ** -24 * want.abs()).all())
    assert ctx.device_status() == binding.SEER_OK
