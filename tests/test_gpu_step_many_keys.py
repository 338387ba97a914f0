"""Steps with more than 8192 compressed keys a unit, or room for them: which are one launch; and the selection of many
candidates, exactly, over the scores that the gate itself reports."""
import numpy as np
import pytest
import torch

import oracle
from paper_2506_08889_b200 import binding, synth
from test_gpu_step_selection import DEV, THETA, scores64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hkv,T,b,L,cap,blocks", [
    (20, 8, 1, 64, 1000, 8200, 8),           # 160 units, short sequences in a large cache
    (6, 8, 1, 64, 200 * 64 - 3, 9000, 160),  # 48 units, 160 tiles each
    (1, 8, 1, 64, 700 * 64, 16384, 600),     # 600 tiles a unit
    (2, 8, 1, 16, 9001 * 16, 9001, 280),     # as many candidates
    (1, 8, 2, 64, 9000 * 64, 9000, 40),      # two query tokens, few units
    (12, 8, 2, 64, 1000, 8200, 8),           # ... and many
])
def test_steps_that_are_one_launch(B, Hkv, T, b, L, cap, blocks, monkeypatch):
    g, d, dg = 2, 128, 64
    seed = 1200 + cap + blocks
    S = -(-L // 64) * 64
    q, qn = (synth.normal_bf16((B, T, Hkv * g, d), seed, x, DEV) for x in ("q", "qn"))
    k, v = (synth.normal_bf16((B, Hkv, S, d), seed, x, DEV) for x in ("k", "v"))
    wq = synth.normal_bf16((Hkv, dg, g * d), seed, "wq", DEV, std=0.02)
    kc = synth.normal_bf16((B, Hkv, cap, dg), seed, "kc", DEV)
    lens_t = torch.full((B,), L, dtype=torch.int32, device=DEV)
    shape, gate, kv = binding.make_shape(B, Hkv * g, Hkv, d, b, 0.09), binding.make_gate(dg, THETA, wq, None, kc, cap), binding.make_kv(k, v, lens_t)
    res = []
    for clusters in ("1", "0"):
        monkeypatch.setenv("SEER_STEP_CLUSTERS", clusters)
        ctx = binding.Context(0)
        idx = torch.full((B, Hkv, blocks), 55, dtype=torch.int32, device=DEV)
        cnt = torch.zeros((B, Hkv), dtype=torch.int32, device=DEV)
        out = torch.empty_like(q)
        before = ctx.launch_count()
        ctx.seer_decode_step_multi(shape, kv, gate, q, qn, T, None, blocks * b, idx, cnt, blocks, out, None)
        res.append((ctx.launch_count() - before, idx.cpu().numpy(), cnt.cpu().numpy(), out.double()))
        assert ctx.device_status() == binding.SEER_OK
    (n1, idx1, cnt1, out1), (n0, idx0, cnt0, out0) = res
    assert n1 == 1 and n0 > 1 and np.array_equal(cnt1, cnt0)
    # where the lists differ, by blocks whose scores are within fp32 rounding of one another
    s = scores64(qn, wq, kc[:, :, :-(-L // b)], L).cpu().numpy()
    same = (idx1 == idx0).all(-1)
    for i, h in zip(*np.nonzero(~same)):
        odd = np.setxor1d(idx1[i, h], idx0[i, h])
        assert np.ptp(s[i, h, odd]) <= 16 * 2.0 ** -24 * 8 * np.abs(s[i, h]).max()
    assert same.mean() > 0.9
    # bf16 outputs from bf16 probabilities, twice
    a, w = out1.view(B, T, Hkv, -1).transpose(1, 2)[torch.as_tensor(same)], out0.view(B, T, Hkv, -1).transpose(1, 2)[torch.as_tensor(same)]
    assert float((a - w).norm() / w.norm()) <= 8e-3


def _kind(kind, n, dg):
    j = torch.arange(n, device=DEV, dtype=torch.float32)
    f = {"smooth": torch.cos(j / 500.0),                       # whole runs of neighbours are taken
         "plateau": torch.where(j % 3 == 0, 1.0 + (j % 128) / 128.0, torch.full_like(j, -300.0)),     # thousands near the top, many equal
         "outlier": torch.where(j == 77, torch.full_like(j, 3.0e4), torch.sin(j * j)),
         "step": (j < n // 2).float(),                         # two values
         "equal": torch.ones_like(j)}[kind]
    u = synth.normal_bf16((dg,), 5, "u", DEV).float()
    return (f[:, None] * u[None, :]).to(torch.bfloat16).expand(1, 1, n, dg).contiguous()


@pytest.mark.parametrize("n", [4097, 6001, 8192])
@pytest.mark.parametrize("kind", ["normal", "smooth", "plateau", "outlier", "step", "equal", "not finite"])
def test_lists_from_the_gate_s_own_scores(n, kind):
    b, d, dg, g = 16, 128, 64, 4
    L = (n + 2) * b + 5                # all n keys are candidates
    qn = synth.normal_bf16((1, g, d), 31, "qn", DEV)
    wq = synth.normal_bf16((1, dg, g * d), 31, "wq", DEV, std=0.02)
    kc = synth.normal_bf16((1, 1, n, dg), 31 + n, "kc", DEV) if kind in ("normal", "not finite") else _kind(kind, n, dg)
    if kind == "not finite":
        kc[:, :, 3::170, 5] = float("inf")
        kc[:, :, 4::190, 9] = -float("inf")
        kc[:, :, 5::230, 2] = float("nan")
    ctx = binding.Context(0)
    lens_t = torch.tensor([L], dtype=torch.int32, device=DEV)
    shape, gate = binding.make_shape(1, g, 1, d, b, 0.09), binding.make_gate(dg, THETA, wq, None, kc, n)
    sc = torch.zeros((1, 1, n + 3), dtype=torch.float32, device=DEV)
    for need in (1, 2, n // 64, n // 32, n // 32 + 1, n // 3, n - 1, n):
        sel = need + 1
        idx = torch.zeros((1, 1, sel), dtype=torch.int32, device=DEV)
        cnt = torch.zeros((1, 1), dtype=torch.int32, device=DEV)
        before = ctx.launch_count()
        ctx.seer_gate_select(shape, gate, lens_t, qn, None, sel * b, idx, cnt, sel, scores_out=sc[:, :, :n])
        assert ctx.launch_count() - before == 1
        s = sc[0, 0, :n].cpu().numpy().astype(np.float64)
        key = np.where(np.isnan(s), -np.inf, s) + 0.0
        # score descending, NaN last, block ascending; then the last block
        order = np.lexsort((np.arange(n), np.isnan(s), -key))
        want = np.append(np.sort(order[:need]), -(-L // b) - 1)
        assert np.array_equal(idx[0, 0].cpu().numpy(), want), (need, kind)
        assert int(cnt) == sel
    assert ctx.device_status() == binding.SEER_OK
