"""A first sweep whose graph cannot be instantiated (GPU).  The failure is a
fake: the library's objects are linked once more with cudaGraphInstantiate
wrapped by a function that returns an error code while a flag is set."""
import ctypes
import os
import subprocess

import pytest
import torch

from paper_2504_10118_gb300 import magpie
from tests.test_gpu_group import Member, orders

pytestmark = pytest.mark.gpu

FAKE = """
#include <cuda_runtime_api.h>
extern "C" {
int fake_instantiate_fails = 0, fake_instantiate_calls = 0;
cudaError_t __real_cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long);
cudaError_t __wrap_cudaGraphInstantiate(cudaGraphExec_t* exec, cudaGraph_t graph, unsigned long long flags) {
  ++fake_instantiate_calls;
  return fake_instantiate_fails ? cudaErrorMemoryAllocation : __real_cudaGraphInstantiate(exec, graph, flags);
}
}
"""


@pytest.fixture(scope="module")
def faked(tmp_path_factory):
    """The library with the wrapped call, in place of the ordinary one."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    magpie.build()
    objs = [os.path.join(magpie.BUILD_DIR, os.path.basename(s) + ".o") for s in magpie.SOURCES]
    if not all(os.path.exists(o) for o in objs):
        magpie.build(force=True)
    d = tmp_path_factory.mktemp("faked")
    src, path = d / "fake.cpp", str(d / "libmagpie_faked.so")
    src.write_text(FAKE)
    subprocess.run(["nvcc", *magpie.ARCH, "-shared", "-Xcompiler", "-fPIC", "-Xlinker", "--wrap=cudaGraphInstantiate",
                    "-o", path, str(src), *objs], check=True)
    with pytest.MonkeyPatch.context() as mp:
        mp.setattr(magpie, "LIB_PATH", path)
        mp.setattr(magpie, "_lib", None)
        magpie.lib()
        yield ctypes.CDLL(path)


@pytest.mark.parametrize("spec", [(75, 32, 5, 9, 1, 2, 8), (201, 128, 3, 23, 3, 3, 4)])
def test_failed_capture_is_no_error_of_the_sweep_that_ran(faked, spec):
    fails = ctypes.c_int.in_dll(faked, "fake_instantiate_fails")
    calls = ctypes.c_int.in_dll(faked, "fake_instantiate_calls")
    mb = Member(spec, 5)
    plain = mb.ctx()
    z_plain = mb.zt
    ctx = mb.ctx()
    z = mb.zt
    out = torch.empty((mb.n, mb.n), dtype=torch.complex64).pin_memory()
    for sweep in range(6):
        o = orders([mb], sweep)[0]
        magpie.magpie_sweep(plain, o)
        before = calls.value
        fails.value = int(sweep < 3)
        try:
            if sweep == 1:
                magpie.magpie_sweep_host(ctx, o.cpu(), None, out)
                assert torch.equal(out, z_plain.cpu())
            else:
                magpie.magpie_sweep(ctx, o)
        finally:
            fails.value = 0
        # tried until it succeeds, once
        assert calls.value - before == (1 if sweep <= 3 else 0)
        assert torch.equal(z, z_plain)
    magpie.magpie_sync(ctx)
    ctx.close()
    plain.close()


@pytest.mark.parametrize("warm", [False, True])
def test_no_sweep_on_a_stream_that_is_captured(warm):
    """Refused with an error, the object untouched, the context usable after."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    magpie.build()
    mb = Member((75, 32, 5, 9, 1, 2, 8), 6)
    plain = mb.ctx()
    z_plain = mb.zt
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        ctx = mb.ctx()
        z = mb.zt
        o = orders([mb], 0)[0]
        if warm:
            magpie.magpie_sweep(ctx, o)
        stream.synchronize()
        before = z.clone()
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        graph.capture_begin()
        with pytest.raises(magpie.MagpieError) as ei:
            magpie.magpie_sweep(ctx, o)
        try:
            graph.capture_end()
        except RuntimeError:
            pass  # the refused call may have invalidated the capture
        assert ei.value.code == magpie.ECUDA
        stream.synchronize()
        assert torch.equal(z, before)
        magpie.magpie_sweep(ctx, o)
        stream.synchronize()
    for _ in range(1 + warm):
        magpie.magpie_sweep(plain, o)
    torch.cuda.synchronize()
    assert torch.equal(z, z_plain)
    ctx.close()
    plain.close()
