"""The gate without a context takes the form that a context's gate call takes under the same switches, and so gives the same
bits; the two forms agree to within fp32 rounding."""
import numpy as np
import pytest
import torch

from paper_2506_08889_b200 import binding, synth
from test_gpu_step_selection import DEV, THETA

pytestmark = pytest.mark.gpu


def _scores(static, n=900, need=40):
    Hkv, g, d, dg, b = 2, 5, 128, 128, 64
    qn = synth.normal_bf16((1, Hkv * g, d), 77, "qn", DEV)
    wq = synth.normal_bf16((Hkv, dg, g * d), 77, "wq", DEV, std=0.02)
    kc = synth.normal_bf16((1, Hkv, n, dg), 77, "kc", DEV)
    lens_t = torch.tensor([n * b - 3], dtype=torch.int32, device=DEV)
    idx, cnt = torch.zeros((1, Hkv, need), dtype=torch.int32, device=DEV), torch.zeros((1, Hkv), dtype=torch.int32, device=DEV)
    sc = torch.zeros((1, Hkv, n), dtype=torch.float32, device=DEV)
    shape, gate = binding.make_shape(1, Hkv * g, Hkv, d, b, 0.09), binding.make_gate(dg, THETA, wq, None, kc, n)
    if static:
        binding.seer_gate_select_static(0, shape, gate, lens_t, qn, need * b, idx, cnt, need, scores_out=sc)
    else:
        binding.Context(0).seer_gate_select(shape, gate, lens_t, qn, None, need * b, idx, cnt, need, scores_out=sc)
    torch.cuda.synchronize()
    return sc[0, :, :n - 1].cpu().numpy(), idx.cpu().numpy()


@pytest.mark.parametrize("switch", [None, ("SEER_STEP_CLUSTERS", "1"), ("SEER_STEP_CLUSTERS", "0"), ("SEER_GATE_WIDEN", "2")])
def test_static_gate_goes_by_the_switches(switch, monkeypatch):
    for name in ("SEER_STEP_CLUSTERS", "SEER_GATE_WIDEN"):
        monkeypatch.delenv(name, raising=False)
    default, _ = _scores(False)
    if switch:
        monkeypatch.setenv(*switch)
    (a, ia), (b, ib) = _scores(True), _scores(False)
    assert np.array_equal(a.view(np.uint32), b.view(np.uint32)) and np.array_equal(ia, ib)
    # sums of 128 products of the size of the scores, each rounded to 2^-24 at most a few times, on either side
    assert np.abs(a - default).max() <= 2 * 8 * 2.0 ** -24 * np.sqrt(128) * np.abs(default).max()
