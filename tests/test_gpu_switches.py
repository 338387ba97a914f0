"""Which kernels a call takes under the environment's switches: by default short calls are one launch; a switch that chooses
among the forms of the other kernels is never passed over without a word."""
import numpy as np
import pytest
import torch

from paper_2506_08889_b200 import binding, synth
from util import bits, check_attention, kernels_of, make_qkv, ref_dense

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
SWITCHES = ("SEER_STEP_CLUSTERS", "SEER_DECODE_WIDE_VARIANT", "SEER_STEP_LIST_FLAGS", "SEER_GATE_WIDEN", "SEER_DECODE_POOL_DIV",
            "SEER_DECODE_MIN_TILES")
ALL = {"gate", "sparse", "dense", "sparse_wide", "step", "step_multi", "step_wide"}


@pytest.mark.parametrize("switch,value,chain", [
    (None, None, set()),
    ("SEER_STEP_CLUSTERS", "1", set()),
    ("SEER_STEP_CLUSTERS", "0", ALL),
    ("SEER_DECODE_WIDE_VARIANT", "8", {"sparse_wide", "step_wide"}),
    ("SEER_DECODE_WIDE_VARIANT", "16", {"sparse_wide", "step_wide"}),
    ("SEER_STEP_LIST_FLAGS", "0", {"step"}),
    ("SEER_STEP_LIST_FLAGS", "1", {"step"}),
    ("SEER_GATE_WIDEN", "2", {"gate", "step", "step_multi", "step_wide"}),
    ("SEER_DECODE_POOL_DIV", "0", ALL - {"gate"}),
    ("SEER_DECODE_MIN_TILES", "4", ALL - {"gate"}),
])
def test_calls_take_the_kernels_that_a_switch_is_about(monkeypatch, switch, value, chain):
    for name in SWITCHES:
        monkeypatch.delenv(name, raising=False)
    if switch:
        monkeypatch.setenv(switch, value)
    B, Hq, Hkv, d, dg, b, S, n = 2, 10, 2, 128, 128, 64, 2048, 8
    q1, k, v = make_qkv(B, Hq, Hkv, S, d, 31, DEV)
    q4 = synth.normal_bf16((B, 4, Hq, d), 31, "q4", DEV)
    q2 = q4[:, :2].contiguous()
    wq = synth.normal_bf16((Hkv, dg, Hq // Hkv * d), 31, "wq", DEV, std=0.02)
    kc = synth.normal_bf16((B, Hkv, S // b, dg), 31, "kc", DEV)
    lens = torch.as_tensor(np.array([S, S - 100], np.int32), device=DEV)
    shape, gate = binding.make_shape(B, Hq, Hkv, d, b, 0.1), binding.make_gate(dg, 1.0e6, wq, None, kc, S // b)
    kv = binding.make_kv(k, v, lens)
    idx = torch.zeros((B, Hkv, n), dtype=torch.int32, device=DEV)
    cnt = torch.zeros((B, Hkv), dtype=torch.int32, device=DEV)
    c = binding.Context(0)
    try:
        calls = {
            "gate": lambda: c.seer_gate_select(shape, gate, lens, q1, None, n * b, idx, cnt, n),
            "sparse": lambda: c.seer_sparse_decode(shape, kv, q1, idx, cnt, n, torch.empty_like(q1)),
            "dense": lambda: c.seer_dense_decode(shape, kv, q1, torch.empty_like(q1)),
            "sparse_wide": lambda: c.seer_sparse_decode_multi(shape, kv, q4, 4, idx, cnt, n, torch.empty_like(q4)),
            "step": lambda: c.seer_decode_step(shape, kv, gate, q1, q1, None, n * b, idx, cnt, n, torch.empty_like(q1), None),
            "step_multi": lambda: c.seer_decode_step_multi(shape, kv, gate, q2, q2, 2, None, n * b, idx, cnt, n, torch.empty_like(q2), None),
            "step_wide": lambda: c.seer_decode_step_multi(shape, kv, gate, q4, q4, 4, None, n * b, idx, cnt, n, torch.empty_like(q4), None),
        }
        for name, call in calls.items():
            call()
            took = kernels_of(call)
            assert took, "no kernel seen"
            if name not in chain:
                want = ["step_cluster_kernel"]
            else:                                           # (the part of a step that the switch is not about may be either)
                gate_part = "gate_cluster_kernel" if switch in ("SEER_STEP_CLUSTERS", "SEER_GATE_WIDEN") else "_cluster_kernel"
                attention_part = "_kernel" if switch == "SEER_GATE_WIDEN" else "decode_kernel"
                want = [gate_part] if name == "gate" else [gate_part, attention_part] if "step" in name else [attention_part]
            assert len(took) == len(want) and all(w in t for w, t in zip(want, took)), (name, took)
        assert c.device_status() == binding.SEER_OK
    finally:
        c.close()


@pytest.mark.parametrize("kind,B,tiles,clusters", [
    # two hundred units of one CTA each: 18 tiles a CTA for lists and dense calls, 64 for a step
    ("sparse", 25, 18, True), ("sparse", 25, 19, False), ("dense", 25, 18, True), ("dense", 25, 19, False),
    ("step", 25, 64, True), ("step", 25, 65, False),
    # sixty-four units of four CTAs: 24
    ("sparse", 8, 96, True), ("sparse", 8, 97, False),
])
def test_lines_between_the_one_launch_form_and_the_decode_kernel(kind, B, tiles, clusters):
    # one long sequence among short ones, which is what the lines are there for; both sides against the oracle
    Hq, Hkv, d, dg, b = 16, 8, 128, 64, 64
    S = tiles * b
    lens = np.array([S - 5] + [(64, 1, 200, 0)[i % 4] for i in range(B - 1)], np.int32)
    q, k, v = make_qkv(B, Hq, Hkv, S, d, 32, DEV)
    wq = synth.normal_bf16((Hkv, dg, Hq // Hkv * d), 32, "wq", DEV, std=0.02)
    kc = synth.normal_bf16((B, Hkv, tiles, dg), 32, "kc", DEV)
    lens_t = torch.as_tensor(lens, device=DEV)
    shape, gate, kv = binding.make_shape(B, Hq, Hkv, d, b, 0.1), binding.make_gate(dg, 1.0e6, wq, None, kc, tiles), binding.make_kv(k, v, lens_t)
    n = -(-lens // b)
    idx = torch.as_tensor(np.where(np.arange(tiles) < n[:, None, None], np.arange(tiles), -1).astype(np.int32).repeat(Hkv, 1), device=DEV)
    cnt = torch.as_tensor(n.astype(np.int32)[:, None].repeat(Hkv, 1), device=DEV)
    out = torch.full((B, Hq, d), float("nan"), dtype=torch.bfloat16, device=DEV)
    lse = torch.full((B, Hq), float("nan"), dtype=torch.float32, device=DEV)
    c = binding.Context(0)
    try:
        call = {"sparse": lambda: c.seer_sparse_decode(shape, kv, q, idx, cnt, tiles, out, lse),
                "dense": lambda: c.seer_dense_decode(shape, kv, q, out, lse),
                "step": lambda: c.seer_decode_step(shape, kv, gate, q, q, None, tiles * b, idx, cnt, tiles, out, lse)}[kind]
        call()
        torch.cuda.synchronize()
        check_attention(out, lse, *ref_dense(bits(q), bits(k), bits(v), lens, 0.1), what=kind)
        took = kernels_of(call)
        assert "decode_kernel" not in took[-1] if clusters else "decode_kernel" in took[-1], took
        assert c.device_status() == binding.SEER_OK
    finally:
        c.close()
