"""CTAs of a recurrence step: as many as the chip holds, wherever the kernel has that many tasks."""
import ctypes as C

import pytest

pytestmark = pytest.mark.gpu


# tasks of the plain kernel: 128 lanes of 2 (FP64) or 4 (FP32) probes, the lanes beyond a row's probes on more rows.
# Four of its CTAs fit an SM (128 registers of 128 threads), 608 a chip of 152.
@pytest.mark.parametrize("n_atoms,n_orb,s,fp64,plain,tasks", [
    (300, 1, 1024, True, False, 1200), (300, 1, 520, True, False, 900), (300, 1, 1024, False, False, 600),
    (100, 1, 4096, False, False, 800), (300, 1, 256, True, False, 300), (300, 1, 32, True, False, 38),
    (5, 1, 4, True, False, 1), (20000, 1, 512, True, False, 40000),
    (400, 9, 388, False, True, 400), (700, 9, 1024, True, True, 2800),
])
def test_plain_kernel_fills_the_chip(n_atoms, n_orb, s, fp64, plain, tasks):
    import torch
    from paper_1812_05264_gb300 import _lib as L, api
    ctx = api.Context()
    H = L.tbk_bsr(n_atoms, n_orb, 7 * n_atoms, None, None, None)
    n = C.c_int32()
    flags = (L.TBK_FP64 if fp64 else 0) | (L.TBK_PLAIN_KERNEL if plain else 0)
    L.call("tbk_test_step_grid", ctx.handle, C.byref(H), s, 20, flags, C.byref(n))
    held = 4 * torch.cuda.get_device_properties(0).multi_processor_count
    assert min(tasks, held) <= n.value <= max(1, tasks)


# 128-probe tasks of the tensor-core step, on a grid of at least one CTA per SM where there are as many
@pytest.mark.parametrize("n_atoms,s", [(100, 512), (40, 1024), (1, 128)])
def test_tensor_core_step_fills_the_chip(n_atoms, s):
    import torch
    from paper_1812_05264_gb300 import _lib as L, api
    ctx = api.Context()
    H = L.tbk_bsr(n_atoms, 9, 13 * n_atoms, None, None, None)
    n = C.c_int32()
    L.call("tbk_test_step_grid", ctx.handle, C.byref(H), s, 20, L.TBK_TENSOR_CORES, C.byref(n))
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    tasks = n_atoms * s // 128
    assert min(tasks, 2 * sms) <= n.value <= tasks
