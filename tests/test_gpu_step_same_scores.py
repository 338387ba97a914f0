"""The one-launch gate's scores do not depend on how many CTAs share a unit: a sequence's are the same bits alone and in a
batch of any size, and so are a step's lists.  And gate queries next to the largest fp32 number stay finite."""
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


@pytest.mark.parametrize("n,T,dg", [(5, 1, 128), (21, 1, 128), (63, 1, 64), (300, 3, 256)])
def test_what_lies_behind_the_candidates_has_no_part(n, T, dg):
    Hkv, g, d, b, cap = 2, 4, 128, 64, n + 23
    L = n * b - 3                      # candidates: the first n - 1 (n - 2) blocks of a cache of n + 23
    wq = synth.normal_bf16((Hkv, dg, g * d), n, "wq", DEV, std=0.02)
    qn = synth.normal_bf16((1, T, Hkv * g, d), n, "qn", DEV)
    kc = synth.normal_bf16((1, Hkv, cap, dg), n, "kc", DEV)
    lens_t = torch.tensor([L], dtype=torch.int32, device=DEV)
    ctx, got = binding.Context(0), []
    m = n - 1 - (T > 1)
    for behind in (0.0, float("nan"), float("inf"), None):
        c = kc.clone()
        if behind is None:
            c = c[:, :, :m + 1].contiguous()         # ... or the cache ends there
        else:
            c[:, :, m:] = behind
        idx, cnt = torch.zeros((1, Hkv, 4), dtype=torch.int32, device=DEV), torch.zeros((1, Hkv), dtype=torch.int32, device=DEV)
        sc = torch.zeros((1, Hkv, c.shape[2]), dtype=torch.float32, device=DEV)
        shape, gate = binding.make_shape(1, Hkv * g, Hkv, d, b, 0.09), binding.make_gate(dg, THETA, wq, None, c, c.shape[2])
        ctx.seer_gate_select_multi(shape, gate, lens_t, qn, None, T, 4 * b, idx, cnt, 4, scores_out=sc)
        got.append(sc[0, :, :m].cpu().numpy().view(np.uint32))
    for other in got[1:]:
        assert np.array_equal(got[0], other)
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


@pytest.mark.parametrize("Hkv,g,T,dg,n,finite", [(2, 4, 1, 128, 4097, True), (8, 5, 1, 128, 2000, False), (2, 4, 1, 256, 700, False),
                                                 (2, 8, 3, 128, 2050, True), (2, 8, 3, 64, 1000, False), (1, 8, 8, 128, 900, False)])
def test_a_step_has_the_gate_s_lists(Hkv, g, T, dg, n, finite):
    # (up to 64 rows: 8 and 16 warps a CTA, one and two clusters a unit, beside the gate's own form)
    d, b, need = 128, 64, 50
    L, seed = n * b - 3, 1600 + n
    qn, q = (synth.normal_bf16((1, T, Hkv * g, d), seed, x, DEV) for x in ("qn", "q"))
    wq = synth.normal_bf16((Hkv, dg, g * d), seed, "wq", DEV, std=0.02)
    kc = synth.normal_bf16((1, Hkv, n, dg), seed, "kc", DEV)
    if not finite:
        kc[:, :, 3::170, 5] = float("inf")
        kc[:, :, 4::190, 9] = -float("inf")
        kc[:, :, 5::23, 2] = float("nan")
    # every third block twice: equal scores, so that one bit more or less would change the list
    kc[:, :, 1:n - 1:3] = kc[:, :, 0:n - 2:3]
    k = synth.normal_bf16((1, Hkv, n * b, d), seed, "k", DEV)
    lens_t = torch.tensor([L], dtype=torch.int32, device=DEV)
    shape, gate, kv = binding.make_shape(1, Hkv * g, Hkv, d, b, 0.09), binding.make_gate(dg, THETA, wq, None, kc, n), binding.make_kv(k, k, lens_t)
    ctx, lists = binding.Context(0), []
    for step in (False, True):
        idx, cnt = torch.zeros((1, Hkv, need), dtype=torch.int32, device=DEV), torch.zeros((1, Hkv), dtype=torch.int32, device=DEV)
        before = ctx.launch_count()
        if step:
            ctx.seer_decode_step_multi(shape, kv, gate, q, qn, T, None, need * b, idx, cnt, need, torch.empty_like(q), None)
        else:
            ctx.seer_gate_select_multi(shape, gate, lens_t, qn, None, T, need * b, idx, cnt, need)
        assert ctx.launch_count() - before == 1
        lists.append(idx.cpu().numpy())
    assert np.array_equal(*lists)
    assert ctx.device_status() == binding.SEER_OK
