"""Which kernels a call takes: clusters up to their lines, one launch or two, and never where a switch of the environment is set
that chooses among the other kernels.  The kernels' names come from the profiler's activity records; a process of its own takes
them, all at once (this file run as a program)."""
import json
import os
import re
import subprocess
import sys

import numpy as np
import pytest
import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path[:0] = [ROOT, os.path.join(ROOT, "tests")]

from paper_2506_08889_b200 import binding, synth  # noqa: E402
from util import bits, check_attention, make_qkv, ref_dense  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
SWITCHES = ("SEER_STEP_CLUSTERS", "SEER_DECODE_WIDE_VARIANT", "SEER_STEP_LIST_FLAGS", "SEER_GATE_WIDEN", "SEER_DECODE_POOL_DIV",
            "SEER_DECODE_MIN_TILES")
CALLS = ("gate", "sparse", "dense", "sparse_rows15", "sparse_wide", "step", "step_multi", "step_wide")
ATTENTION = set(CALLS) - {"gate"}
SETTINGS = [                              # a switch, its value, the calls that do not take the one-launch form then
    (None, None, set()),
    ("SEER_STEP_CLUSTERS", "1", set()),
    ("SEER_STEP_CLUSTERS", "0", set(CALLS)),
    ("SEER_DECODE_WIDE_VARIANT", "8", {"sparse_wide", "step_wide"}),
    ("SEER_DECODE_WIDE_VARIANT", "16", {"sparse_wide", "step_wide"}),
    ("SEER_STEP_LIST_FLAGS", "0", {"step"}),
    ("SEER_STEP_LIST_FLAGS", "1", {"step"}),
    ("SEER_GATE_WIDEN", "2", {"gate", "step", "step_multi", "step_wide"}),
    ("SEER_DECODE_POOL_DIV", "0", ATTENTION),
    ("SEER_DECODE_MIN_TILES", "4", ATTENTION),
]
EVEN, DEALT, DECODE, STEP, GATE = "list_step_cluster_kernel", "dealt_decode_kernel", "decode_kernel", "step_cluster_kernel", "gate_cluster_kernel"
SMALL_WS = 3_600_000                      # bytes: the decode kernel's partials of 200 units, not the dealt lists'
LINES = [                                 # a call, its sequences, the tiles of its one long list, its kernels (, block, workspace)
    # two hundred units of one CTA each: above 22 tiles lists may be dealt, above 128 the decode kernel; a step is one launch up
    # to 64, and from there to 128 the dealing kernel follows
    ("sparse", 25, 22, [EVEN]), ("sparse", 25, 23, [DEALT]), ("dense", 25, 22, [EVEN]), ("dense", 25, 23, [DEALT]),
    ("dense", 25, 128, [DEALT]), ("dense", 25, 129, [DECODE]),
    ("step", 25, 64, [STEP]), ("step", 25, 65, [STEP, DEALT]), ("step", 25, 128, [STEP, DEALT]), ("step", 25, 129, [GATE, DECODE]),
    # 304 units: more than there are places
    ("sparse", 38, 4, [DECODE]), ("dense", 38, 4, [DECODE]),
    # sixty-four units of four CTAs
    ("sparse", 8, 96, [EVEN]), ("sparse", 8, 97, [DEALT]), ("dense", 8, 512, [DEALT]), ("dense", 8, 513, [DECODE]),
    # eight of sixteen: up to 32 tiles a CTA a cluster per unit; the heads of one sequence have lists as long, which are not dealt
    ("dense", 1, 512, [EVEN]), ("dense", 1, 769, [DEALT]),
    ("step", 1, 1024, [STEP]), ("step", 1, 1025, [STEP]), ("step", 1, 2049, [GATE, DECODE]),
    # blocks of 16 tokens: 256 numbers a CTA
    ("step", 25, 64, [STEP], 16), ("step", 25, 65, [GATE, DECODE], 16),
    # partial results that do not fit
    ("sparse", 25, 22, [EVEN], 64, SMALL_WS), ("sparse", 25, 23, [DECODE], 64, SMALL_WS), ("step", 25, 65, [GATE, DECODE], 64, SMALL_WS),
]


def _switch_calls(c):
    B, Hq, Hkv, d, dg, b, S, n = 2, 10, 2, 128, 128, 64, 2048, 8
    q1, k, v = make_qkv(B, Hq, Hkv, S, d, 31, DEV)
    q4 = synth.normal_bf16((B, 4, Hq, d), 31, "q4", DEV)
    q2, q3 = q4[:, :2].contiguous(), q4[:, :3].contiguous()
    wq = synth.normal_bf16((Hkv, dg, Hq // Hkv * d), 31, "wq", DEV, std=0.02)
    kc = synth.normal_bf16((B, Hkv, S // b, dg), 31, "kc", DEV)
    lens = torch.as_tensor(np.array([S, S - 100], np.int32), device=DEV)
    shape, gate = binding.make_shape(B, Hq, Hkv, d, b, 0.1), binding.make_gate(dg, 1.0e6, wq, None, kc, S // b)
    kv = binding.make_kv(k, v, lens)
    idx = torch.zeros((B, Hkv, n), dtype=torch.int32, device=DEV)
    cnt = torch.zeros((B, Hkv), dtype=torch.int32, device=DEV)
    return {
        "gate": lambda: c.seer_gate_select(shape, gate, lens, q1, None, n * b, idx, cnt, n),
        "sparse": lambda: c.seer_sparse_decode(shape, kv, q1, idx, cnt, n, torch.empty_like(q1)),
        "dense": lambda: c.seer_dense_decode(shape, kv, q1, torch.empty_like(q1)),
        "sparse_rows15": lambda: c.seer_sparse_decode_multi(shape, kv, q3, 3, idx, cnt, n, torch.empty_like(q3)),
        "sparse_wide": lambda: c.seer_sparse_decode_multi(shape, kv, q4, 4, idx, cnt, n, torch.empty_like(q4)),
        "step": lambda: c.seer_decode_step(shape, kv, gate, q1, q1, None, n * b, idx, cnt, n, torch.empty_like(q1), None),
        "step_multi": lambda: c.seer_decode_step_multi(shape, kv, gate, q2, q2, 2, None, n * b, idx, cnt, n, torch.empty_like(q2), None),
        "step_wide": lambda: c.seer_decode_step_multi(shape, kv, gate, q4, q4, 4, None, n * b, idx, cnt, n, torch.empty_like(q4), None),
    }


def _line_call(c, kind, B, tiles, b=64):
    """One long sequence among short ones, every block listed: the call, and its output to be checked."""
    Hq, Hkv, d, dg = 16, 8, 128, 64
    S = tiles * 64
    blocks = S // b
    lens = np.array([S - 5] + [(64, 1, 200, 0)[i % 4] for i in range(B - 1)], np.int32)
    q, k, v = make_qkv(B, Hq, Hkv, S, d, 32, DEV)
    wq = synth.normal_bf16((Hkv, dg, Hq // Hkv * d), 32, "wq", DEV, std=0.02)
    kc = synth.normal_bf16((B, Hkv, blocks, dg), 32, "kc", DEV)
    lens_t = torch.as_tensor(lens, device=DEV)
    shape, gate, kv = binding.make_shape(B, Hq, Hkv, d, b, 0.1), binding.make_gate(dg, 1.0e6, wq, None, kc, blocks), binding.make_kv(k, v, lens_t)
    n = -(-lens // b)
    idx = torch.as_tensor(np.where(np.arange(blocks) < n[:, None, None], np.arange(blocks), -1).astype(np.int32).repeat(Hkv, 1), device=DEV)
    cnt = torch.as_tensor(n.astype(np.int32)[:, None].repeat(Hkv, 1), device=DEV)
    out = torch.full((B, Hq, d), float("nan"), dtype=torch.bfloat16, device=DEV)
    lse = torch.full((B, Hq), float("nan"), dtype=torch.float32, device=DEV)
    call = {"sparse": lambda: c.seer_sparse_decode(shape, kv, q, idx, cnt, blocks, out, lse),
            "dense": lambda: c.seer_dense_decode(shape, kv, q, out, lse),
            "step": lambda: c.seer_decode_step(shape, kv, gate, q, q, None, S, idx, cnt, blocks, out, lse)}[kind]
    return call, lambda: check_attention(out, lse, *ref_dense(bits(q), bits(k), bits(v), lens, 0.1), what=kind)


def _kernels_of(call):
    from torch.autograd import DeviceType
    from torch.profiler import ProfilerActivity, profile
    call()
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA], acc_events=True) as prof:
        call()
        torch.cuda.synchronize()
    found = sorted((e.time_range.start, e.name) for e in prof.events() if e.device_type == DeviceType.CUDA)
    return [name for _, name in found if "seer" in name and "kernel" in name]


def _name(kernel):
    """A kernel's own name, without its scope and parameters."""
    return re.search(r"(\w+_kernel)\b", kernel).group(1)


def _main():
    seen = {"switches": [], "lines": []}
    for switch, value, _ in SETTINGS:
        for name in SWITCHES:
            os.environ.pop(name, None)
        if switch:
            os.environ[switch] = value                      # read when a context is created
        c = binding.Context(0)
        seen["switches"].append({name: _kernels_of(call) for name, call in _switch_calls(c).items()})
        c.close()
    for name in SWITCHES:
        os.environ.pop(name, None)
    for kind, B, tiles, _, *more in LINES:
        c = binding.Context(0, *more[1:])
        seen["lines"].append(_kernels_of(_line_call(c, kind, B, tiles, *more[:1])[0]))
        c.close()
    print(json.dumps(seen))


@pytest.fixture(scope="module")
def seen():
    done = subprocess.run([sys.executable, os.path.abspath(__file__)], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert done.returncode == 0, done.stderr[-2000:]
    found = json.loads(done.stdout.strip().splitlines()[-1])
    if not any(found["lines"]):
        pytest.skip("no activity records here")
    return found


@pytest.mark.parametrize("at", range(len(SETTINGS)), ids=["%s-%s" % s[:2] for s in SETTINGS])
def test_calls_take_the_kernels_that_a_switch_is_about(seen, at):
    switch, value, chain = SETTINGS[at]
    for name, took in seen["switches"][at].items():
        if name not in chain:
            want = [EVEN if name in ("sparse", "dense") else STEP]
            took = [_name(t) for t in took]
        else:
            # (the part of a step that the switch is not about may be either; decode_kernel<sparse, paged, tiles of rows,
            # small blocks, tensor memory>)
            gate = "gate_cluster_kernel" if switch in ("SEER_STEP_CLUSTERS", "SEER_GATE_WIDEN") else "_cluster_kernel"
            rows = "8, false, false" if value == "8" else "8, false, true" if "wide" in name else "2, false, false" if name[-2:] in ("15", "ti") else "1, false, false"
            attention = "_kernel" if switch == "SEER_GATE_WIDEN" else "decode_kernel<%s, false, %s>" % ("false" if name == "dense" else "true", rows)
            want = [gate] if name == "gate" else [gate, attention] if "step" in name else [attention]
        assert len(took) == len(want) and all(w in t for w, t in zip(want, took)), (name, want, took)


@pytest.mark.parametrize("at", range(len(LINES)), ids=["-".join(str(x) for x in (*l[:3], *l[4:])) for l in LINES])
def test_lines_between_the_forms(seen, at):
    kind, B, tiles, kernels, *more = LINES[at]
    assert [_name(t) for t in seen["lines"][at]] == kernels, seen["lines"][at]
    c = binding.Context(0, *more[1:])
    try:
        call, check = _line_call(c, kind, B, tiles, *more[:1])
        call()
        torch.cuda.synchronize()
        check()
        assert c.device_status() == binding.SEER_OK
    finally:
        c.close()


if __name__ == "__main__":
    _main()
