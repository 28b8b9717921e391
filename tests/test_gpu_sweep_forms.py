"""Every way to run a sweep takes the same kernels (GPU): a context's first
sweep, the replayed ones, the profiled and the host-fed ones.  Where
deterministic = 0 takes the ordered update (minibatches of small windows of up
to 65536 pixels, windows of 128 and more) that shows in the bits of the object."""
import numpy as np
import pytest
import torch

from paper_2504_10118_gb300 import magpie, synth
from tests.test_gpu_group import Member, orders

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    magpie.build()
    magpie.lib()


def ctx_of(mb, deterministic):
    dev = torch.device("cuda")
    z = torch.from_numpy(mb.z0.astype(np.complex64)).to(dev)
    p = magpie.magpie_params_of(mb.n, mb.n, mb.m, mb.N, mb.L, mb.B, 0.1, deterministic=deterministic)
    ctx = magpie.magpie_create(p, z, torch.from_numpy(mb.Q.astype(np.complex64)).to(dev), torch.from_numpy(mb.pos).to(dev),
                               torch.from_numpy(mb.d.astype(np.float32)).to(dev))
    return ctx, z


# (n, m, grid, step, jitter, levels, minibatch): dozens of windows over most pixels
SPECS = [(61, 16, 8, 5, 1, 3, 32), (75, 32, 8, 6, 1, 2, 32), (179, 128, 6, 9, 2, 3, 12)]


@pytest.mark.parametrize("spec", SPECS)
def test_every_sweep_takes_the_sweeps_kernels(spec):
    mb = Member(spec, 21)
    ordered, z_ordered = ctx_of(mb, 1)
    fast, z_fast = ctx_of(mb, 0)
    intensities = torch.from_numpy(mb.d.astype(np.float32)).pin_memory()
    calls = ["sweep", "sweep", "profile", "host", "host_async", "sweep"]
    for i, call in enumerate(calls):
        o = orders([mb], i)[0]
        magpie.magpie_sweep(ordered, o)
        if call == "sweep":
            magpie.magpie_sweep(fast, o)
        elif call == "profile":
            magpie.magpie_profile_sweep(fast, o)
        elif call == "host":
            magpie.magpie_sweep_host(fast, o.cpu(), intensities)
        else:
            magpie.magpie_sweep_host_async(fast, o.cpu().pin_memory(), intensities)
            magpie.magpie_sync(fast)
        torch.cuda.synchronize()
        assert torch.equal(z_ordered, z_fast), (i, call)
    ordered.close()
    fast.close()


# (m, levels, minibatch, update_probe): whether steps of deterministic = 0 use the float atomics
MEMORY = [(128, 3, 8, 0, False), (256, 5, 2, 0, False), (64, 3, 8, 0, False), (64, 3, 64, 0, True), (64, 3, 128, 0, True),
          (64, 5, 8, 0, True), (128, 3, 8, 1, True), (128, 6, 8, 0, True), (32, 2, 8, 0, True)]


@pytest.mark.parametrize("m,levels,minibatch,probe,atomic", MEMORY)
def test_accumulators_are_held_where_steps_use_them(m, levels, minibatch, probe, atomic):
    """Device memory that deterministic = 0 adds to a context on 3000 x 3000
    pixels: 16 bytes per pixel (137 MiB) or nothing, to allocation granularity."""
    n, N = 3000, 128
    dev = torch.device("cuda")
    z = torch.ones((n, n), dtype=torch.complex64, device=dev)
    Q = torch.from_numpy(synth.make_probe(m).astype(np.complex64)).to(dev)
    pos = torch.from_numpy(np.random.default_rng(m).integers(0, n - m + 1, (N, 2)).astype(np.int32)).to(dev)
    d = magpie.magpie_forward_intensities(z, Q, pos, m)

    def used(deterministic):
        p = magpie.magpie_params_of(n, n, m, N, levels, minibatch, 0.1, probe, 0.1, deterministic)
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        ctx = magpie.magpie_create(p, z, Q, pos, d)
        taken = before - torch.cuda.mem_get_info()[0]
        magpie.magpie_step(ctx, torch.arange(8 if minibatch > 8 else minibatch, dtype=torch.int32, device=dev))
        magpie.magpie_sync(ctx)
        ctx.close()
        return taken

    used(1)  # whatever the first context of a side leaves behind
    extra = used(0) - used(1)
    granule = 2 << 20
    assert abs(extra - (16 * n * n if atomic else 0)) <= 4 * granule, extra
