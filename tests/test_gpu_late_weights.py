"""Gate weights that the kernel launched just before a call writes, and writes late: it lets its dependents start at once,
as a kernel with programmatic launch may, and stores some 30 us later.  A call must not read its weights before that
kernel has completed."""
import numpy as np
import pytest
import torch

from paper_2506_08889_b200 import binding, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
THETA = 1.0e6

LATE_COPY = r"""
extern "C" __global__ void late_copy(uint4* dst, const uint4* src, int n16) {
    asm volatile("griddepcontrol.launch_dependents;");
    for (int k = 0; k < 30; ++k) __nanosleep(1000);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n16; i += gridDim.x * blockDim.x) dst[i] = src[i];
}
"""


@pytest.fixture(scope="module")
def late_copy():
    kernel = torch.cuda._compile_kernel(LATE_COPY, "late_copy")

    def run(dst, src):
        assert dst.is_contiguous() and src.is_contiguous() and dst.numel() == src.numel() and dst.numel() % 8 == 0
        kernel(grid=(16, 1, 1), block=(256, 1, 1), args=[dst, src, dst.numel() // 8])

    return run


@pytest.mark.parametrize("b,dg", [(16, 128), (32, 64), (64, 128), (128, 128), (64, 256)])
def test_build(ctx, late_copy, b, dg):
    B, Hkv, S, d = 2, 8, 2048, 128
    kn = synth.normal_bf16((B, Hkv, S, d), 71, "kn", DEV)
    wk = synth.normal_bf16((Hkv, dg, 3 * d), 71, "wk", DEV, std=0.02)
    shape = binding.make_shape(B, 2 * Hkv, Hkv, d, b, 0.1)
    lens = torch.as_tensor(np.array([S, S - 300], np.int32), device=DEV)
    got = []
    for late in (False, True):
        w = torch.zeros_like(wk) if late else wk
        kc = torch.zeros((B, Hkv, S // b, dg), dtype=torch.bfloat16, device=DEV)
        gate = binding.make_gate(dg, THETA, None, w, kc, S // b)
        torch.cuda.synchronize()
        if late:
            late_copy(w, wk)
        ctx.seer_kcomp_append(shape, gate, lens, kn, first_block=0, num_blocks=S // b)
        torch.cuda.synchronize()
        got.append(kc)
    assert torch.equal(*got) and got[0].any()
    assert ctx.device_status() == binding.SEER_OK


@pytest.mark.parametrize("n,T,dg", [(300, 1, 128), (300, 3, 64), (4000, 1, 256), (9000, 1, 128)])
def test_gate_and_step(ctx, late_copy, n, T, dg):
    B, Hq, Hkv, d, b, max_sel = 2, 16, 4, 128, 16, 20
    lens = torch.as_tensor(np.array([n * b, n * b // 2 + 5], np.int32), device=DEV)
    q, qn = (synth.normal_bf16((B, T, Hq, d), 72, x, DEV) for x in ("q", "qn"))
    k, v = (synth.normal_bf16((B, Hkv, n * b, d), 72, x, DEV) for x in ("k", "v"))
    kn = synth.normal_bf16((B, Hkv, b, d), 72, "kn", DEV)
    wq = synth.normal_bf16((Hkv, dg, Hq // Hkv * d), 72, "wq", DEV, std=0.02)
    wk = synth.normal_bf16((Hkv, dg, 3 * d), 72, "wk", DEV, std=0.02)
    kc0 = synth.normal_bf16((B, Hkv, n, dg), 72, "kc", DEV)
    shape = binding.make_shape(B, Hq, Hkv, d, b, 0.0884)
    kv = binding.make_kv(k, v, lens)
    for step in (False, True):
        got = []
        for late in (False, True):
            w = torch.zeros(wq.numel() + wk.numel(), dtype=torch.bfloat16, device=DEV)
            wq_in, wk_in = w[:wq.numel()].view(wq.shape), w[wq.numel():].view(wk.shape)
            kc = kc0.clone()
            gate = binding.make_gate(dg, THETA, wq_in, wk_in, kc, n)
            idx = torch.zeros((B, Hkv, max_sel), dtype=torch.int32, device=DEV)
            cnt = torch.zeros((B, Hkv), dtype=torch.int32, device=DEV)
            out = torch.zeros((B, T, Hq, d), dtype=torch.bfloat16, device=DEV)
            both = torch.cat([wq.flatten(), wk.flatten()])
            if not late:
                w.copy_(both)
            torch.cuda.synchronize()
            if late:
                late_copy(w, both)
            if step:
                ctx.seer_decode_step_multi(shape, kv, gate, q, qn, T, kn, max_sel * b, idx, cnt, max_sel, out, None, rows_block_local=True)
            else:
                ctx.seer_gate_select_multi(shape, gate, lens, qn, None, T, max_sel * b, idx, cnt, max_sel)
            torch.cuda.synchronize()
            got.append((idx, cnt, out, kc))
        for x, y in zip(*got):
            assert torch.equal(x, y)
        assert (got[0][3] != kc0).any() == step and got[0][0].any()
    assert ctx.device_status() == binding.SEER_OK
