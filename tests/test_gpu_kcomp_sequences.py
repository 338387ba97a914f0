"""The bulk build's two ways to add up the sequences' blocks (up to 32 sequences, every warp for itself; more, the CTA
together), with sequences that have no complete block, and its two ways to cut the runs: within a head where the heads
divide the CTAs (3, 4, 5 and 8 heads do: the last CTAs stay away) and across heads where they do not (20 and 32)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2506_08889_b200 import binding, synth
from util import bits, kc_tolerance

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("B,Hkv,b,dg", [(31, 4, 64, 128), (32, 8, 16, 128), (33, 8, 64, 64), (32, 5, 128, 128), (40, 3, 32, 128),
                                             (31, 20, 64, 128), (40, 32, 32, 64)])
def test_build_of_many_sequences(B, Hkv, b, dg):
    lens = np.array([(i * 37 % 11) * b + (i * 13) % b for i in range(B)], np.int32)
    S, d = 12 * b, 128
    kn = synth.normal_bf16((B, Hkv, S, d), 91, "kn", DEV)
    wk = synth.normal_bf16((Hkv, dg, 3 * d), 91, "wk", DEV, std=0.02)
    kc = torch.full((B, Hkv, 12, dg), 7.0, dtype=torch.bfloat16, device=DEV)
    lens_t = torch.as_tensor(lens, device=DEV)
    ctx = binding.Context(0)
    for _ in range(2):
        ctx.seer_kcomp_append(binding.make_shape(B, Hkv, Hkv, d, b, 0.1), binding.make_gate(dg, 1.0e6, None, wk, kc, 12), lens_t, kn,
                              first_block=0, num_blocks=12)
    torch.cuda.synchronize()
    _, want = oracle.kcomp(bits(kn), bits(wk), b, 0, 12, 12, 1.0e6)
    out = kc.to(torch.float64).cpu().numpy()
    for i, L in enumerate(lens):
        n = int(L) // b
        assert np.all(out[i, :, n:] == 7.0), i
        if n:
            assert np.all(np.abs(out[i, :, :n] - want[i, :, :n]) <= kc_tolerance(want[i, :, :n])), i
    assert ctx.device_status() == binding.SEER_OK
