"""Context lengths and page tables that the preceding kernel writes while the decode is already
resident.  A small kernel lets its dependents start at once, holds back a short bounded time and only
then writes them; the decode and its merge, launched behind it, have planned from what stood there
before.  The results are, bit for bit, those of a call on settled inputs, and what stood there
before is not reported."""

import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from tests.test_gpu_flat_batches import _batch

pytestmark = pytest.mark.gpu

SOURCE = r"""
// One CTA.  The wait is bounded: 300 sleeps of at most about 0.2 us each.
__global__ void late(int* ctx, const int* ctx_src, int n, int* table, const int* table_src, int m) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    for (int i = 0; i < 300; ++i) __nanosleep(100);
    for (int i = threadIdx.x; i < n; i += blockDim.x) ctx[i] = ctx_src[i];
    for (int i = threadIdx.x; i < m; i += blockDim.x) table[i] = table_src[i];
}
extern "C" int launch_late(void* ctx, const void* ctx_src, int n, void* table, const void* table_src, int m, void* stream) {
    late<<<1, 256, 0, (cudaStream_t)stream>>>((int*)ctx, (const int*)ctx_src, n, (int*)table, (const int*)table_src, m);
    return (int)cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def late(tmp_path_factory):
    from paper_2607_28699_gb300 import build
    d = tmp_path_factory.mktemp("late")
    (d / "late.cu").write_text(SOURCE)
    subprocess.run([build._nvcc(), *build.ARCH, "-O2", "-shared", "-Xcompiler", "-fPIC", "-o", str(d / "late.so"),
                    str(d / "late.cu")], check=True)
    f = ctypes.CDLL(os.path.join(str(d), "late.so")).launch_late
    f.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p]
    return f


def _lens(batch, longest):
    rng = np.random.default_rng(batch)
    lens = [int(x) for x in rng.integers(1, longest, batch)]
    lens[0] = longest
    if batch > 2:
        lens[1] = 0
    return lens


# one sequence (split plan), flattened with hints in decode and merge (<= 32), in the decode only
# (<= 512), in neither; a short table (split plan)
@pytest.mark.parametrize("batch,longest", [(1, 2400), (2, 2400), (5, 3000), (32, 1200), (33, 700), (513, 700), (16, 300)])
@pytest.mark.parametrize("scheme,bits", [("int8", 8), ("int8", 10), ("g32", 8), ("fp8", 8)])
def test_late_inputs(late, batch, longest, scheme, bits):
    import paper_2607_28699_gb300 as wc
    code = {"int8": wc.SCHEME_DITHER_INT8, "g32": wc.SCHEME_DITHER_INT8_G32, "fp8": wc.SCHEME_FP8_E4M3}[scheme]
    lens = _lens(batch, longest)
    desc, table, ctx, q, cache = _batch(lens, code, 16, 4, bits=bits)
    ws = wc.Workspace(desc, batch, table.shape[1])
    want = [x.clone() for x in wc.metered_decode_attention(desc, 0, q, table, ctx, cache, ws)]
    torch.cuda.synchronize()
    assert wc.read_status(ws) == 0
    full, low = torch.full_like(ctx, longest), torch.zeros_like(ctx)
    rng = torch.Generator().manual_seed(batch)
    stale = [low, full, torch.full_like(ctx, -7), torch.full_like(ctx, 1 << 30),
             torch.randint(0, longest + 1, (batch,), generator=rng).int().cuda(), ctx.flip(0).contiguous(), ctx.clone()]
    bad_table = torch.where(torch.rand(table.shape, generator=rng).cuda() < 0.5, torch.full_like(table, -3),
                            torch.full_like(table, 1 << 30))
    outs = [torch.empty_like(x) for x in want]
    stream = torch.cuda.current_stream().cuda_stream
    for before in stale:
        for table_before in (bad_table, table):
            live_ctx, live_table = before.clone(), table_before.clone()
            for x in outs:
                x.fill_(float("nan"))
            torch.cuda.synchronize()
            assert late(live_ctx.data_ptr(), ctx.data_ptr(), batch, live_table.data_ptr(), table.data_ptr(), table.numel(),
                        stream) == 0
            wc.metered_decode_attention(desc, 0, q, live_table, live_ctx, cache, ws, *outs)
            torch.cuda.synchronize()
            assert wc.read_status(ws) == 0
            for x, y in zip(outs, want):
                assert torch.equal(x, y)


def test_late_inputs_in_a_captured_step(late):
    import paper_2607_28699_gb300 as wc
    lens = [2400, 900, 2000, 16]
    desc, table, ctx, q, cache = _batch(lens, wc.SCHEME_DITHER_INT8, 16, 4)
    ws = wc.Workspace(desc, 4, table.shape[1])
    outs = [torch.empty_like(x) for x in wc.metered_decode_attention(desc, 0, q, table, ctx, cache, ws)]
    src = ctx.clone()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        stream = torch.cuda.current_stream().cuda_stream
        for _ in range(20):
            assert late(ctx.data_ptr(), src.data_ptr(), 4, table.data_ptr(), table.data_ptr(), 0, stream) == 0
            wc.metered_decode_attention(desc, 0, q, table, ctx, cache, ws, *outs)
    want = wc.metered_decode_attention(desc, 0, q, table, src, cache, wc.Workspace(desc, 4, table.shape[1]))
    for lens_before in ([0, 0, 0, 0], [2400, 2400, 2400, 2400], [16, 2000, 900, 2400]):
        ctx.copy_(torch.tensor(lens_before, dtype=torch.int32))
        graph.replay()
        torch.cuda.synchronize()
        assert wc.read_status(ws) == 0
        for x, y in zip(outs, want):
            assert torch.equal(x, y)
