"""The split form of the window phase (windows of 64 and more, three kernels
over strips of 16 lines) against the cluster kernel, bit for bit: a context
swept by itself takes the split form, the persistent form of a group always
takes the cluster kernel, which the parity tests hold to the oracle."""
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


# (n, m, grid, step, jitter, minibatch): odd object sides, a short last minibatch
SIDES = {64: (131, 64, 4, 17, 2, 6), 128: (201, 128, 3, 23, 3, 4), 256: (301, 256, 2, 29, 3, 3)}


@pytest.mark.parametrize("m,levels", [(m, L) for m in SIDES for L in range(1, (5 if m == 64 else 6) + 1)])
def test_split_form_equals_cluster_kernel(m, levels):
    """Every level count, the deepest of which falls back to the cluster kernel."""
    n, m, g, s, j, B = SIDES[m]
    mb = Member((n, m, g, s, j, levels, B), 7 + levels)
    alone = mb.ctx()
    z_alone = mb.zt
    member = mb.ctx()
    z_member = mb.zt
    group = magpie.magpie_group_create([member])
    magpie.magpie_group_set_persistent(group, 1)
    for sweep in range(2):
        o = orders([mb], sweep)
        magpie.magpie_sweep(alone, o[0])
        magpie.magpie_group_sweep(group, o)
    assert magpie.magpie_group_status(group) == magpie.OK
    assert torch.equal(z_alone, z_member)
    a, b = magpie.magpie_window_values(alone), magpie.magpie_window_values(member)
    for x, y in zip(a, b):  # FP64 sums of FP32 warp sums, the pixels split over warps in another way
        assert float(((x - y) / y).abs().max()) < 256 * 2.0 ** -24
    group.close()
    alone.close()
    member.close()


def test_skipped_index_and_raw_intensities():
    """An index out of range leaves its window out and is reported; a host
    sweep that reads the intensities in the window phase gives the sweep's bits."""
    n, m, g, s, j, B = SIDES[64]
    mb = Member((n, m, g, s, j, 3, B), 3)
    good, bad = mb.ctx(), None
    z_good = mb.zt
    bad = mb.ctx()
    z_bad = mb.zt
    idx = torch.tensor([0, 5, 9], dtype=torch.int32, device="cuda")
    magpie.magpie_step(good, idx)
    magpie.magpie_step(bad, torch.tensor([0, mb.N, 5, -1, 9], dtype=torch.int32, device="cuda"))
    with pytest.raises(magpie.MagpieError) as ei:
        magpie.magpie_window_values(bad)
    assert ei.value.code == magpie.EINDEX
    assert torch.equal(z_good, z_bad)
    host = mb.ctx()
    z_host = mb.zt
    plain = mb.ctx()
    z_plain = mb.zt
    order = synth.make_order(mb.N, 1)
    magpie.magpie_sweep_host_async(host, torch.from_numpy(order).pin_memory(),
                                   torch.from_numpy(mb.d.astype(np.float32)).pin_memory())
    magpie.magpie_sync(host)
    magpie.magpie_sweep(plain, torch.from_numpy(order).cuda())
    torch.cuda.synchronize()
    # sqrt(d) by the same rounding in both places
    assert torch.equal(z_host, z_plain)
    for c in (good, bad, host, plain):
        c.close()


@pytest.mark.parametrize("n,step", [(645, 50), (897, 70)])
def test_large_update_tiles_and_atomics(n, step):
    """Objects large enough for 760 tiles of 32 x 16 or of 32 x 32 are updated in
    those, a group forced to 16 x 16 tiles gives the same bits; the float
    atomics that m = 64 keeps for minibatches of 64 and more agree to rounding."""
    mb = Member((n, 64, 12, step, 5, 3, 64), 5)
    alone = mb.ctx()
    z_alone = mb.zt
    member = mb.ctx()
    z_member = mb.zt
    dev = torch.device("cuda")
    z_atomic = torch.from_numpy(mb.z0.astype(np.complex64)).to(dev)
    p = magpie.magpie_params_of(mb.n, mb.n, mb.m, mb.N, mb.L, mb.B, 0.1, deterministic=0)
    atomic = magpie.magpie_create(p, z_atomic, torch.from_numpy(mb.Q.astype(np.complex64)).to(dev),
                                  torch.from_numpy(mb.pos).to(dev), torch.from_numpy(mb.d.astype(np.float32)).to(dev))
    group = magpie.magpie_group_create([member])
    magpie.magpie_group_set_persistent(group, 0)
    magpie.magpie_group_set_apply_shape(group, 0)
    o = orders([mb], 0)
    magpie.magpie_sweep(alone, o[0])
    magpie.magpie_sweep(atomic, o[0])
    magpie.magpie_group_sweep(group, o)
    torch.cuda.synchronize()
    assert torch.equal(z_alone, z_member)
    # at most 64 windows per pixel and step, three steps: sums in another order
    d = (z_alone - z_atomic).abs().max() / z_alone.abs().max()
    assert float(d) < 3 * 64 * 2.0 ** -24
    group.close()
    for c in (alone, member, atomic):
        c.close()
