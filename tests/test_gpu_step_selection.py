"""The one-launch step's lists where its selection changes form: candidates in registers (up to sixteen a thread), a histogram
over all of them, the short list of many candidates, 16 worker warps above 8192 keys, crowded bins; and scores that are not
finite, which leave the matrix instructions for plain products."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2506_08889_b200 import binding, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
THETA = 1.0e6


def rope64(y, pos):
    half = y.shape[-1] // 2
    ang = pos * THETA ** (-2.0 * torch.arange(half, device=DEV, dtype=torch.float64) / y.shape[-1])
    a, d = y[..., :half], y[..., half:]
    return torch.cat([a * ang.cos() - d * ang.sin(), d * ang.cos() + a * ang.sin()], -1)


def scores64(qn, wq, kc, L):
    """[B, Hkv, n]: the largest over the query tokens of the gate's scores, in 64 bits."""
    T, Hkv = qn.shape[1], wq.shape[0]
    x = qn.view(qn.shape[0], T, Hkv, -1).double()
    y = torch.einsum("bthn,hcn->bthc", x, wq.double())
    y = torch.stack([rope64(y[:, t], L - T + t) for t in range(T)], 1)
    return torch.einsum("bhnc,bthc->bthn", kc.double(), y).amax(1) / math.sqrt(wq.shape[1])


@pytest.mark.parametrize("Hkv,g,T,dg,b,n,need,kind", [
    (2, 4, 1, 128, 16, 1025, 40, ""),          # 1024 candidates: four a thread
    (2, 4, 1, 128, 16, 1026, 40, ""),          # 1025: eight
    (1, 5, 1, 64, 16, 2049, 700, ""),          # 2048
    (1, 5, 1, 256, 16, 2050, 700, ""),         # 2049: sixteen
    (2, 8, 1, 128, 32, 4096, 100, ""),         # 4095: as before; 4097: the short list
    (2, 8, 1, 128, 32, 4098, 127, ""),
    (2, 8, 1, 128, 32, 4098, 129, ""),         # too many places for it: the histogram over all
    (1, 4, 1, 128, 16, 8190, 60, "crowded"),   # a far outlier: neither list helps
    (1, 4, 1, 128, 16, 8194, 200, ""),         # 16 worker warps
    (1, 4, 1, 64, 16, 16384, 300, ""),         # the most keys
    (1, 4, 1, 128, 16, 16384, 2000, "ties"),
    (2, 8, 3, 128, 64, 2050, 33, ""),          # 24 rows: 16 worker warps
    (1, 8, 8, 64, 64, 4100, 30, ""),           # 64 rows: two clusters a unit
])
def test_lists_against_64_bit_scores(Hkv, g, T, dg, b, n, need, kind):
    Hq, d, L = Hkv * g, 128, n * b - 3
    seed = 700 + n + need
    q, qn = (synth.normal_bf16((1, T, Hq, d), seed, x, DEV) for x in ("q", "qn"))
    k = synth.normal_bf16((1, Hkv, n * b, d), seed, "k", DEV)
    wq = synth.normal_bf16((Hkv, dg, g * d), seed, "wq", DEV, std=0.02)
    kc = synth.normal_bf16((1, Hkv, n, dg), seed, "kc", DEV)
    if kind == "crowded":
        kc[:, :, 7] *= 1e4
    elif kind == "ties":
        kc = kc[:, :, torch.arange(n, device=DEV) % 7].contiguous()
    forced = n - (L - T) // b
    sel = need + forced
    ctx = binding.Context(0)
    shape, gate = binding.make_shape(1, Hq, Hkv, d, b, 0.09), binding.make_gate(dg, THETA, wq, None, kc, n)
    lens_t = torch.tensor([L], dtype=torch.int32, device=DEV)
    kv = binding.make_kv(k, k, lens_t)
    idx = torch.full((1, Hkv, sel + 5), 55, dtype=torch.int32, device=DEV)
    cnt = torch.zeros((1, Hkv), dtype=torch.int32, device=DEV)
    out = torch.empty((1, T, Hq, d), dtype=torch.bfloat16, device=DEV)
    before = ctx.launch_count()
    for _ in range(4):                         # (one right behind the other)
        if T == 1:
            ctx.seer_decode_step(shape, kv, gate, q[:, 0], qn[:, 0], None, sel * b, idx, cnt, sel + 5, out[:, 0], None)
        else:
            ctx.seer_decode_step_multi(shape, kv, gate, q, qn, T, None, sel * b, idx, cnt, sel + 5, out, None)
    assert ctx.launch_count() - before == 4
    torch.cuda.synchronize()
    assert ctx.device_status() == binding.SEER_OK
    s = scores64(qn, wq, kc, L)[0, :, :n - forced].cpu().numpy()
    idx, cnt = idx[0].cpu().numpy(), cnt[0].cpu().numpy()
    for h in range(Hkv):
        got = idx[h, :sel]
        assert cnt[h] == sel and np.all(np.diff(got) > 0) and np.all(idx[h, sel:] == -1)
        assert np.array_equal(got[need:], np.arange(n - forced, n))
        if kind == "ties":                     # equal keys have equal scores: the lower block first
            want = np.sort(np.lexsort((np.arange(n - forced), -np.round(s[h], 6)))[:need])
            assert np.array_equal(got[:need], want)
            continue
        # a block within fp32 rounding of the last one taken may fall on either side: a sum of d_gate products of the size
        # of the scores, each rounded to 2^-24 at most a few times
        # (the outlier's own products have no part in another block's score)
        eps = 8 * 2.0 ** -24 * math.sqrt(dg) * np.abs(np.delete(s[h], 7) if kind == "crowded" else s[h]).max()
        last = np.sort(s[h])[::-1][need - 1]
        taken = np.zeros(n - forced, bool)
        taken[got[:need]] = True
        assert np.all(s[h][taken] >= last - eps) and np.all(s[h][~taken] <= last + eps)


@pytest.mark.parametrize("T,dg", [(1, 64), (1, 128), (1, 256), (4, 128)])
def test_scores_that_are_not_finite(T, dg):
    # one infinite channel of a key gives plus or minus infinity, two that disagree NaN, as plain products do
    Hkv, g, d, b, n = 2, 4, 128, 64, 300
    qn = synth.normal_bf16((1, T, Hkv * g, d), 71, "qn", DEV)
    wq = synth.normal_bf16((Hkv, dg, g * d), 71, "wq", DEV, std=0.02)
    kc = synth.normal_bf16((1, Hkv, n, dg), 71, "kc", DEV)
    kc[:, :, 3::17, 5] = float("inf")
    kc[:, :, 4::19, 9] = -float("inf")
    kc[:, :, 5::23, 2] = float("nan")
    kc[:, :, 100, :2] = 3.0e38
    L = n * b - 3
    ctx = binding.Context(0)
    lens_t = torch.tensor([L], dtype=torch.int32, device=DEV)
    idx = torch.zeros((1, Hkv, 40), dtype=torch.int32, device=DEV)
    cnt = torch.zeros((1, Hkv), dtype=torch.int32, device=DEV)
    sc = torch.zeros((1, Hkv, n), dtype=torch.float32, device=DEV)
    shape, gate = binding.make_shape(1, Hkv * g, Hkv, d, b, 0.09), binding.make_gate(dg, THETA, wq, None, kc, n)
    ctx.seer_gate_select_multi(shape, gate, lens_t, qn, None, T, 40 * b, idx, cnt, 40, scores_out=sc)
    torch.cuda.synchronize()
    # (the largest over the query tokens passes a NaN by)
    y = torch.stack([scores64(qn[:, t:t + 1], wq, kc, L - T + 1 + t) for t in range(T)])
    want = torch.where(torch.isnan(y), -math.inf, y).amax(0) if T > 1 else y[0]
    got, want = sc[0, :, :n - 1].cpu().numpy(), want[0, :, :n - 1].float().cpu().numpy()
    ok = np.isfinite(want)
    assert np.array_equal(np.isnan(got), np.isnan(want)) and np.array_equal(got[np.isinf(want)], want[np.isinf(want)])
    assert np.allclose(got[ok], want[ok], rtol=2e-5, atol=1e-5)
    want_idx, want_cnt = oracle.select_multi(sc.cpu().numpy(), np.array([L], np.int32), b, 40 * b, T, 40)
    assert np.array_equal(idx.cpu().numpy(), want_idx) and np.array_equal(cnt.cpu().numpy(), want_cnt)
    assert ctx.device_status() == binding.SEER_OK
