"""Steps of more than 64 and up to 128 tiles a CTA: two launches, of which the first does even lists and the second, where they
are uneven, the attention; batches on both sides of that line, a block that has just filled among them, every width of the gate,
the one launch of a single sequence and the chain of blocks of 16 tokens, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2506_08889_b200 import binding, synth
from util import bits, check_attention, make_qkv, ref_sparse, to_paged

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
SCALE, THETA = 0.0884, 1.0e6

EVEN, UNEVEN = [5120 - 64 * (x % 5) - 7 * (x % 3) for x in range(25)], [640] * 12 + [5120] + [64 * x for x in range(12)]
CASES = [
    # Hq, Hkv, b, page, cached tokens, budget in blocks, d_gate, launches, lists uneven (tiles a CTA by 0.46 us above what all take and 8 us)
    (32, 8, 64, 0, EVEN, 72, 128, 2, False),                                                                       # 200 units, a CTA each
    (16, 8, 64, 0, UNEVEN, 72, 128, 2, True),                                                                      # one long sequence, an empty one
    (40, 8, 32, 64, [10432, 10048] + [128 + 32 * x for x in range(8)], 300, 128, 2, True),                         # 80 units, clusters of 2, two long
    (8, 2, 128, 0, [16384 + 128 * x for x in range(40)], 100, 128, 2, False),                                      # 80 units, two tiles a block
    (16, 8, 64, 0, EVEN, 72, 256, 2, False),
    (16, 8, 32, 0, UNEVEN, 144, 256, 2, True),
    (16, 8, 32, 64, EVEN, 150, 64, 2, False),
    (8, 8, 64, 0, UNEVEN, 75, 64, 2, True),
    (16, 8, 64, 0, [70400 - 5], 1030, 128, 1, False),                                                              # one sequence: its heads' lists are as long
    (16, 8, 16, 0, EVEN, 280, 128, 3, False),                                                                      # more numbers than a CTA holds
]


def _uneven(lens, b, budget, Hkv, S):
    """The rule that both launches go by."""
    tiles = [min(-(-L // b), budget) * b / 64 if b >= 64 else -(-min(-(-L // b), budget) * b // 64) for L in lens]
    total, most, units = sum(tiles) * Hkv, max(tiles), len(lens) * Hkv
    return 0.46 * most / S > max(0.004 * total, 0.46 * total / (units * S)) + 8


@pytest.mark.parametrize("case", range(len(CASES)))
def test_step_of_long_lists(ctx, case):
    Hq, Hkv, b, page, lens, budget, dg, want_launches, uneven = CASES[case]
    B, d, seed = len(lens), 128, 700 + case
    if want_launches == 2:
        assert _uneven(lens, b, budget, Hkv, 1 if B * Hkv > 148 else 2) == uneven
    unit = max(page, b, 64)
    cap = -(-max(lens) // unit) * unit
    nb = cap // b
    lens = np.array(lens, np.int32)
    q, k, v = make_qkv(B, Hq, Hkv, cap, d, seed, DEV)
    for i in range(B):
        v[i, :, lens[i]:] = float("nan")
    qn = synth.normal_bf16((B, Hq, d), seed, "qn", DEV)
    wq = synth.normal_bf16((Hkv, dg, Hq // Hkv * d), seed, "wq", DEV, std=0.02)
    wk = synth.normal_bf16((Hkv, dg, 3 * d), seed, "wk", DEV, std=0.02)
    kc = synth.normal_bf16((B, Hkv, nb, dg), seed, "kc", DEV)
    window = synth.normal_bf16((B, Hkv, b, d), seed, "win", DEV)
    shape = binding.make_shape(B, Hq, Hkv, d, b, SCALE)
    lens_t = torch.as_tensor(lens, device=DEV)
    if page:
        kp, vp, table = to_paged(k, v, page, seed)
        kv = binding.make_kv(kp, vp, lens_t, max_seq_len=cap, page_table=table, page_size=page)
    else:
        kv = binding.make_kv(k, v, lens_t)
    gate = binding.make_gate(dg, THETA, wq, wk, kc.clone(), nb)
    want_kc = kc.clone()
    ctx.seer_kcomp_append(shape, binding.make_gate(dg, THETA, wq, wk, want_kc, nb), lens_t, window, rows_block_local=True, first_block=-1)
    sc = torch.zeros((B, Hkv, nb), dtype=torch.float32, device=DEV)
    idx0, cnt0 = (torch.full(s, 55, dtype=torch.int32, device=DEV) for s in ((B, Hkv, budget), (B, Hkv)))
    ctx.seer_gate_select(shape, binding.make_gate(dg, THETA, wq, wk, kc, nb), lens_t, qn, None, budget * b, idx0, cnt0, budget, scores_out=sc)
    torch.cuda.synchronize()
    want_idx, want_cnt = oracle.select(sc.cpu().numpy(), lens, b, budget * b, budget)
    ref = ref_sparse(bits(q), bits(k), bits(torch.nan_to_num(v)), lens, want_idx, want_cnt, b, SCALE)
    for _ in range(3):                                      # (each overlaps the one before)
        got_kc = kc.clone()
        gate = binding.make_gate(dg, THETA, wq, wk, got_kc, nb)
        idx, cnt = torch.full_like(idx0, 55), torch.full_like(cnt0, 55)
        out = torch.full((B, Hq, d), float("nan"), dtype=torch.bfloat16, device=DEV)
        lse = torch.full((B, Hq), float("nan"), device=DEV)
        before = ctx.launch_count()
        ctx.seer_decode_step(shape, kv, gate, q, qn, window, budget * b, idx, cnt, budget, out, lse, rows_block_local=True)
        launches = ctx.launch_count() - before
    torch.cuda.synchronize()
    assert launches == (want_launches if ctx.one_launch else 3)
    assert np.array_equal(cnt.cpu().numpy(), want_cnt) and np.array_equal(idx.cpu().numpy(), want_idx)
    assert torch.equal(got_kc, want_kc)
    check_attention(out, lse, *ref, what=f"case {case}")
    assert ctx.device_status() == binding.SEER_OK
