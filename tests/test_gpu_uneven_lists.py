"""Given lists and dense calls whose lists are so uneven that what long units have above a line is dealt to the clusters that end
before it: units cut anywhere, units without a tile, shares of several units, units of many shares, every cluster size, against
the oracle."""
import numpy as np
import pytest
import torch

from paper_2506_08889_b200 import binding, synth
from util import bits, check_attention, make_qkv, ref_dense, ref_sparse, to_paged

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
SCALE = 0.0884

CASES = [
    # Hq, Hkv, b, page, cached tokens, listed blocks of each sequence (None: dense)
    (32, 8, 64, 0, [5120 - 7, 700, 64, 1, 0] + [300] * 11, [64, 5, 1, 1, 3, 0] + [2, 4, 5, 3, 1, 2, 5, 0, 4, 2]),      # 128 units, clusters of 2
    (4, 1, 64, 0, [57600 - 30, 65, 640], None),                                                                       # 3 units, clusters of 16
    (16, 8, 32, 128, [5120, 4999, 5120] + [512 - x for x in range(22)], [160, 150, 155] + [3 + x % 7 for x in range(22)]),      # 200 units, a CTA each
    (20, 4, 128, 0, [130] * 13 + [8192 - 64] + [1000] * 6, [2] * 13 + [60] + [1, 0, 7, 3, 2, 5]),                      # 80 units, the long one among them
    (8, 2, 16, 64, [9000] * 2 + [50 * x + 1 for x in range(18)], [500, 411] + [x % 9 for x in range(18)]),             # 40 units, four blocks a tile
    (4, 1, 64, 0, [70001], None),                                                                                     # one unit, all other clusters without
    (8, 2, 32, 64, [60000, 300], [1800, 5]),                                                                          # 4 units, two of them long
    (8, 1, 64, 0, [55000, 0, 0, 0, 52000, 63, 64, 65, 0, 128], None),                                                  # shares that begin behind empty units
    (16, 8, 64, 0, [4096 - 7 if x % 11 == 3 else 60 for x in range(24)], None),                                        # 192 units, 24 of them of many shares
    (16, 8, 64, 0, [64 * (1 + x) if x % 7 else 8000 + 64 * x for x in range(18)], None),                           # shares that end near units' ends
]
CLUSTERS = [(2, 128), (16, 3), (1, 200), (2, 80), (4, 40), (16, 16), (16, 16), (16, 10), (1, 192), (2, 144)]      # CTAs each, how many


def _uneven(tiles, S, clusters):
    """The kernel's rule: a CTA alone takes 0.46 us a tile, all together 0.004, a deal 5 us and twelve tiles at least."""
    total, most = sum(tiles), max(tiles)
    return 0.46 * most / S > max(0.004 * total, 0.46 * total / (clusters * S), 0.46 * 12) + 5


@pytest.mark.parametrize("case", range(len(CASES)))
def test_uneven_lists(ctx, case):
    Hq, Hkv, b, page, lens, keep = CASES[case]
    n = [-(-L // 64) for L in lens] if keep is None else [-(-min(k, -(-L // b)) * b // 64) for k, L in zip(keep, lens)]
    assert _uneven([x for x in n for _ in range(Hkv)], *CLUSTERS[case]) and max(n) <= 128 * CLUSTERS[case][0]
    B, d, seed = len(lens), 128, 500 + case
    unit = max(page, b, 64)
    cap = -(-max(lens) // unit) * unit
    lens = np.array(lens, np.int32)
    q, k, v = make_qkv(B, Hq, Hkv, cap, d, seed, DEV, token_major=case == 3)
    for i in range(B):
        v[i, :, lens[i]:] = float("nan")                    # rows past the end may hold anything
    shape = binding.make_shape(B, Hq, Hkv, d, b, SCALE)
    lens_t = torch.as_tensor(lens, device=DEV)
    if page:
        kp, vp, table = to_paged(k, v, page, seed)
        kv = binding.make_kv(kp, vp, lens_t, max_seq_len=cap, page_table=table, page_size=page)
    else:
        kv = binding.make_kv(k, v, lens_t)
    qh, kh, vh = bits(q), bits(k), bits(torch.nan_to_num(v))
    if keep is None:
        ref = ref_dense(qh, kh, vh, lens, SCALE)
        call = lambda o, l: ctx.seer_dense_decode(shape, kv, q, o, l)
    else:
        keep = [min(n, -(-int(L) // b)) for n, L in zip(keep, lens)]
        max_sel = max(keep)
        idx, cnt = synth.random_block_lists([max(int(L), 1) for L in lens], Hkv, b, keep, max_sel, seed)
        ref = ref_sparse(qh, kh, vh, lens, idx, cnt, b, SCALE)
        idx_t, cnt_t = torch.from_numpy(idx).to(DEV), torch.from_numpy(cnt).to(DEV)
        call = lambda o, l: ctx.seer_sparse_decode(shape, kv, q, idx_t, cnt_t, max_sel, o, l)
    outs = [(torch.full((B, Hq, d), float("nan"), dtype=torch.bfloat16, device=DEV), torch.full((B, Hq), float("nan"), device=DEV))
            for _ in range(4)]
    for out, lse in outs:                                   # (each overlaps the one before)
        call(out, lse)
    torch.cuda.synchronize()
    for out, lse in outs:
        check_attention(out, lse, *ref, what=f"case {case}")
        if ctx.one_launch:                                  # the pieces are put together in a fixed order
            assert torch.equal(out, outs[0][0]) and torch.equal(lse, outs[0][1])
    assert ctx.device_status() == binding.SEER_OK


@pytest.mark.parametrize("batch,tiles", [(24, 64), (16, 96)])
def test_one_long_list_among_short_ones_costs_no_more_than_without_clusters(monkeypatch, batch, tiles):
    # (dealt at 8 us a deal it took 1.3 and 1.25 times as long; host-bound runs make both alike)
    Hq, Hkv, d, cap = 32, 8, 128, 64 * tiles
    lens = torch.as_tensor(np.array([cap if i == batch // 2 else 64 for i in range(batch)], np.int32), device=DEV)
    q, k, v = (torch.randn(s, device=DEV, dtype=torch.bfloat16) for s in ((batch, Hq, d), (batch, Hkv, cap, d), (batch, Hkv, cap, d)))
    out, lse = torch.empty_like(q), torch.empty((batch, Hq), device=DEV)
    shape, kv = binding.make_shape(batch, Hq, Hkv, d, 64, SCALE), binding.make_kv(k, v, lens)
    ctxs = []
    for clusters in ("1", "0"):
        monkeypatch.setenv("SEER_STEP_CLUSTERS", clusters)
        ctxs.append(binding.Context(0))
    times = [[], []]
    for _ in range(9):
        for c, t in zip(ctxs, times):
            a, z = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            for i in range(60):
                if i == 10:
                    a.record()
                c.seer_dense_decode(shape, kv, q, out, lse)
            z.record()
            torch.cuda.synchronize()
            t.append(a.elapsed_time(z))
    for c in ctxs:
        c.close()
    assert np.median(times[0]) <= 1.17 * np.median(times[1]), times
