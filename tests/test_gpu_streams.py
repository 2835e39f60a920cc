"""Conventions of the C ABI that the header states beside the arithmetic: calls are capturable in a CUDA graph once
the first call on the device has run, and host threads may call concurrently (each with its own stream, outputs and
workspace).  Every result is also held to the oracle's bound."""
import threading

import numpy as np
import pytest
import torch

from conftest import to_oracle
from plans import gemv_kernel
from oracle import xfp_oracle as xo
import paper_2605_14844_b200 as xfp
from paper_2605_14844_b200 import synth

pytestmark = pytest.mark.gpu

TOL = 1e-3


def _x_dev(x16):
    return torch.from_numpy(x16.view(np.int16)).cuda().view(torch.float16)


def _within_bound(q, x16, y):
    ref, absum = xo.gemv(to_oracle(q), x16)
    got = y.float().cpu().numpy().astype(np.float64)
    assert np.all(np.isfinite(got)) and np.all(np.abs(got - ref) <= TOL * absum + 1e-30)


# the kernel in the operand layout at 1 to 16 rows of x, and (KERNELS_OF, checked below) every other kernel of the dispatch;
# K slices through the workspace (96 x 12288)
CASES = [(0, 4, 200, 1024, 1), (1, 3, 200, 1024, 1), (0, 4, 200, 1024, 2), (1, 4, 200, 1024, 2), (0, 6, 2500, 768, 4),
         (1, 5, 2500, 768, 3), (0, 3, 640, 2048, 8), (1, 4, 640, 2048, 16), (0, 5, 96, 12288, 1), (1, 6, 2500, 768, 8)]
KERNELS_OF = {(0, 4, 200, 1024, 4): "frag", (1, 4, 512, 4096, 1): "lane", (0, 5, 9600, 128, 2): "lane_batch",
              (1, 4, 19200, 512, 12): "gemm", (0, 3, 200, 1024, 2): "pair", (1, 2, 33, 16384, 3): "batch",
              (1, 3, 19000, 512, 2): "v2a", (1, 2, 32, 40960, 3): "generic"}
CASES += list(KERNELS_OF)


@pytest.mark.parametrize("mode,bits,rows,cols,batch", CASES)
def test_calls_are_capturable_in_a_cuda_graph(mode, bits, rows, cols, batch):
    """Three dependent-free calls captured on a side stream and replayed twice give the bits of the eager calls."""
    desc = xfp.XfpDesc(mode, rows, cols, bits, 128, 32 if mode else 0, 32, int(0.01 * rows * cols))
    want = KERNELS_OF.get((mode, bits, rows, cols, batch))
    assert want is None or gemv_kernel(desc, batch) == want
    q = synth.random_quantized(mode, rows, cols, bits, 0.01, seed=9500 + 10 * bits + mode + batch)
    pm = xfp.pack_tensors(q, col_bits=16)
    xs = [synth.activations(batch, cols, seed=9600 + i) for i in range(3)]
    xd = [_x_dev(x) for x in xs]
    eager = [pm.gemv(x).clone() for x in xd]            # the first calls on the device: kernel attributes are set here
    torch.cuda.synchronize()
    ys = [torch.zeros_like(e) for e in eager]
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(side):
        with torch.cuda.graph(g, stream=side):
            for x, y in zip(xd, ys):
                pm.gemv(x, y=y, stream=side)
    for _ in range(2):
        for y in ys:
            y.zero_()
        g.replay()
        torch.cuda.synchronize()
        for e, y in zip(eager, ys):
            assert torch.equal(e, y)
    for x16, y in zip(xs, ys):
        _within_bound(q, x16, y)
    tickets = pm.workspace[: ((rows + 31) // 32) * 4].view(torch.int32)
    assert int(tickets.abs().sum().item()) == 0


def test_host_threads_call_concurrently():
    """Four host threads, each with its own stream, matrix, workspace and outputs, call the library at the same time
    (ctypes releases the interpreter lock during a call): every result equals the one the same call gave alone."""
    specs = [(0, 4, 2500, 768, 1), (1, 3, 640, 2048, 2), (0, 6, 2500, 768, 4), (1, 4, 200, 1024, 8)]
    work = []
    for i, (mode, bits, rows, cols, batch) in enumerate(specs):
        q = synth.random_quantized(mode, rows, cols, bits, 0.01, seed=9700 + i)
        pm = xfp.pack_tensors(q, col_bits=16)
        x16 = synth.activations(batch, cols, seed=9800 + i)
        xd = _x_dev(x16)
        alone = pm.gemv(xd).clone()
        torch.cuda.synchronize()
        _within_bound(q, x16, alone)
        work.append((pm, xd, alone))
    errors = []

    def run(pm, xd, alone):
        try:
            torch.cuda.set_device(0)
            stream = torch.cuda.Stream()
            y = torch.empty_like(alone)
            for _ in range(200):
                pm.gemv(xd, y=y, stream=stream)
            stream.synchronize()
            if not torch.equal(y, alone):
                errors.append("a concurrent call gave other bits")
        except Exception as e:  # reported on the main thread
            errors.append(repr(e))

    threads = [threading.Thread(target=run, args=w) for w in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


LATE = """
#include <cuda_runtime.h>
// releases its dependents at once, then waits and copies
__global__ void late_copy_kernel(const uint4* src, uint4* dst, size_t n, long long clocks) {
    asm volatile("griddepcontrol.launch_dependents;");
    const long long t0 = clock64();
    while (clock64() - t0 < clocks) __nanosleep(1000);
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) dst[i] = src[i];
}
extern "C" int late_copy(const void* src, void* dst, size_t bytes, long long clocks, void* stream) {
    late_copy_kernel<<<8, 256, 0, (cudaStream_t)stream>>>((const uint4*)src, (uint4*)dst, bytes / 16, clocks);
    return cudaGetLastError() != cudaSuccess;
}
"""


@pytest.fixture(scope="module")
def late_copy(tmp_path_factory):
    import ctypes as C
    import subprocess
    from paper_2605_14844_b200 import build as xbuild
    d = tmp_path_factory.mktemp("late")
    (d / "late.cu").write_text(LATE)
    subprocess.run([xbuild.NVCC, *xbuild.FLAGS[:2], "-Xcompiler", "-fPIC", "-shared", str(d / "late.cu"), "-o", str(d / "late.so")],
                   check=True)
    fn = C.CDLL(str(d / "late.so")).late_copy

    def call(src, dst, clocks=400000):
        assert fn(C.c_void_p(src.data_ptr()), C.c_void_p(dst.data_ptr()), C.c_size_t(src.numel()), C.c_longlong(clocks),
                  C.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    return call


@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16])
@pytest.mark.parametrize("mode,rows,cols,m", [(0, 4096, 4096, 100), (1, 2560, 2048, 300), (0, 1024, 1024, 40), (0, 1024, 256, 65)])
def test_prefill_waits_for_a_blob_whose_producer_releases_early(late_copy, mode, rows, cols, m, dtype):
    """The blob is completed by a kernel that lets its dependents start before it has written it.  The GEMV calls exclude that
    (xfp.h); the prefill form reads the blob only when the kernel in front is complete.  Both blobs are without outliers and
    valid, so that a call that read the earlier one would give the earlier matrix's y."""
    old, new = (xfp.pack_tensors(synth.random_quantized_torch(mode, rows, cols, 4, 0.0, 9700 + i, lib_size=32, group_size=128))
                for i in range(2))
    x = torch.randn((m, cols), generator=torch.Generator().manual_seed(9710)).to(dtype).cuda()
    ws = torch.zeros(xfp.xfp_gemm_typed_workspace_size(new.desc, m, dtype), dtype=torch.uint8, device="cuda")
    ref, y = (torch.empty((m, rows), dtype=torch.float32, device="cuda") for _ in range(2))
    xfp.xfp_gemm_typed(new.desc, new.packed, x, ref, ws)
    for _ in range(3):
        blob = old.packed.clone()
        torch.cuda.synchronize()
        late_copy(new.packed, blob)
        xfp.xfp_gemm_typed(new.desc, blob, x, y, ws)
        torch.cuda.synchronize()
        assert torch.equal(y, ref) and int(ws[:4].view(torch.int32).item()) == 0
