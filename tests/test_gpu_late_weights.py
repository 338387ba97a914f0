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


@pytest.fixture(scope="module")
def ctx():
    c = binding.Context(0)
    yield c
    c.close()


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
