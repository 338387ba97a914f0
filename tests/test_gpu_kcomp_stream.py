"""The bulk build of the compressed keys as one streaming kernel, for every block size and from one block on: runs of
blocks that cross sequences and heads, items that end inside a gathered stage, sequences without a complete block, and
the keys whose strides it leaves to the plain kernel."""
import numpy as np
import pytest
import torch

import oracle
from paper_2506_08889_b200 import binding, synth
from util import bits, kc_tolerance

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
THETA = 1.0e6


@pytest.fixture(scope="module")
def ctx():
    c = binding.Context(0)
    yield c
    c.close()


CASES = [
    # Hkv, b, d_gate, lengths, first block, token-major, heads share one set of keys
    (1, 64, 128, [64], 0, False, False),                                # one block in all
    (8, 64, 128, [64 * 41 + 5, 0, 63, 64 * 7], 0, True, False),         # runs within a head
    (3, 128, 64, [128 * 300, 128 * 11 + 127, 128 * 160], 3, False, False),   # 49 CTAs a head, runs of several items
    (7, 128, 128, [128 * 33, 128 * 50 + 1], 0, True, False),
    (100, 64, 128, [64 * 9, 64 * 5 + 9], 0, False, False),              # more heads than divide the CTAs: heads change in a run
    (150, 32, 64, [32 * 7 + 3], 0, False, False),                       # more heads than CTAs
    (5, 32, 128, [32 * 333 + 31, 32, 31], 1, True, False),
    (2, 16, 128, [16 * 1001 + 7, 16 * 3, 0, 16 * 18], 0, False, False),
    (11, 16, 64, [16 * 77, 16 * 21 + 15], 5, True, False),
    (4, 64, 128, [64 * 20], 0, False, True),
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_build(ctx, case):
    Hkv, b, dg, lens, first, token_major, shared = CASES[case]
    B, d, seed = len(lens), 128, 500 + case
    S = max(lens)
    nb = S // b + 2                                          # entries for blocks that do not exist
    if token_major:
        kn = synth.normal_bf16((B, S, Hkv, d), seed, "kn", DEV).permute(0, 2, 1, 3)
    elif shared:
        kn = synth.normal_bf16((B, 1, S, d), seed, "kn", DEV).expand(B, Hkv, S, d)
    else:
        kn = synth.normal_bf16((B, Hkv, S, d), seed, "kn", DEV)
    wk = synth.normal_bf16((Hkv, dg, 3 * d), seed, "wk", DEV, std=0.02)
    shape = binding.make_shape(B, Hkv * 2, Hkv, d, b, 0.1)
    lens_t = torch.as_tensor(np.array(lens, np.int32), device=DEV)
    got = []
    for _ in range(2):
        kc = torch.full((B, Hkv, nb, dg), 7.0, dtype=torch.bfloat16, device=DEV)
        gate = binding.make_gate(dg, THETA, None, wk, kc, nb)
        ctx.seer_kcomp_append(shape, gate, lens_t, kn, first_block=first, num_blocks=nb - first)
        got.append(kc)
    torch.cuda.synchronize()
    assert torch.equal(got[0], got[1])
    n_all = S // b
    _, want = oracle.kcomp(bits(kn[:, :, :n_all * b].contiguous()), bits(wk), b, 0, n_all, n_all, THETA)
    out = got[0].to(torch.float64).cpu().numpy()
    for i, L in enumerate(lens):
        n = L // b
        assert np.all(out[i, :, n:] == 7.0) and np.all(out[i, :, :first] == 7.0)
        if n > first:
            assert np.all(np.abs(out[i, :, first:n] - want[i, :, first:n]) <= kc_tolerance(want[i, :, first:n])), (i, n)
    assert ctx.device_status() == binding.SEER_OK
