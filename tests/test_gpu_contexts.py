"""Two library contexts in one process on two CUDA contexts (two devices, or one device twice): what the library sets per kernel
belongs to a CUDA context and must be set in each."""
import ctypes as C

import numpy as np
import pytest
import torch

import lsp_synth as S
from gpu_util import DEV

pytestmark = pytest.mark.gpu


def test_tensor_core_gemms_in_a_second_cuda_context():
    """The shared-memory limit of a kernel is raised in every CUDA context: the streaming and the paired GEMM after the same calls in
    the first one.  Ones times ones over K = 512: 512 exactly."""
    from paper_2603_05454_b200 import LSPDecoder, SchedCfg
    from paper_2603_05454_b200.binding import ModelCfg, SchedCfgC, WeightsC, lib
    N, K, rows = 256, 512, (100, 300)
    sh = S.ModelShape(1, 64, 1, 1, 64, 64, 128, dtype="bf16")
    dec = LSPDecoder(sh, S.make_weights(sh, 0, device=DEV), SchedCfg(), 1, 8, device=DEV)
    one = lambda m: torch.ones(m, K, dtype=torch.bfloat16, device=DEV)
    for M in rows:
        assert bool((dec.op_linear(0, one(M), one(N), None, torch.empty(M, N, dtype=torch.bfloat16, device=DEV)) == 512).all())
    dec.close()

    cu = C.CDLL("libcuda.so.1")
    ok = lambda rc: rc == 0 or pytest.fail(f"CUDA driver call failed ({rc})")
    ctx, old, handle, bufs = C.c_void_p(), C.c_void_p(), C.c_void_p(), []
    ok(cu.cuCtxCreate_v2(C.byref(ctx), 0, torch.device(DEV).index))           # and makes it current
    try:
        def alloc(n, bf16_bits=0):
            p = C.c_uint64()
            ok(cu.cuMemAlloc_v2(C.byref(p), C.c_size_t(2 * n)))
            ok(cu.cuMemsetD16_v2(p, C.c_ushort(bf16_bits), C.c_size_t(n)))
            bufs.append(p)
            return p.value
        mc = ModelCfg(1, 64, 1, 1, 64, 64, 128, 1e-5, 1e4, 1, 127)
        sc = SchedCfg().to_c()
        ws, kv = lib.lsp_workspace_bytes(C.byref(mc), 1, 8), lib.lsp_kv_cache_bytes(C.byref(mc), 1, 8)
        z = alloc(64 * 192)
        per_layer = (C.c_void_p * 1)(z)
        wc = WeightsC(z, z, z, *[C.cast(per_layer, C.POINTER(C.c_void_p))] * 7)
        assert lib.lsp_init(C.byref(handle), C.byref(mc), C.byref(sc), C.byref(wc), alloc(kv // 2), alloc((ws + 1) // 2), ws, 1, 8, None) == 0
        A, W, out = alloc(max(rows) * K, 0x3F80), alloc(N * K, 0x3F80), alloc(max(rows) * N)
        for M in rows:
            rc = lib.lsp_op_linear(handle, 0, A, W, None, out, M, N, K)
            assert rc == 0, lib.lsp_last_error(handle).decode()
            got = np.zeros((M, N), dtype=np.uint16)
            ok(cu.cuMemcpyDtoH_v2(got.ctypes.data_as(C.c_void_p), C.c_uint64(out), C.c_size_t(got.nbytes)))
            assert (got == 0x4400).all()
    finally:
        if handle:
            lib.lsp_destroy(handle)
        for p in bufs:
            cu.cuMemFree_v2(p)
        cu.cuCtxPopCurrent_v2(C.byref(old))
        cu.cuCtxDestroy_v2(ctx)
    assert float(one(2).sum()) == 2 * K                                       # the first context goes on as before
