"""Steps of which no window index is in range (GPU): every window is skipped,
so the object stays as it is, bit for bit, whatever the steps before left in
the context's buffers, and the next valid step is that of a context that never
saw the invalid one.  For every form whose kernels overlap their predecessors."""
import pytest
import torch

from paper_2504_10118_gb300 import magpie
from tests.test_gpu_group import Member, orders

pytestmark = pytest.mark.gpu

# (n, m, grid, step, jitter, minibatch): the strip kernels' three window sides and a small one
SIDES = {32: (101, 32, 4, 21, 2, 5), 64: (131, 64, 4, 17, 2, 6), 128: (201, 128, 3, 23, 3, 4), 256: (301, 256, 2, 29, 3, 3)}
ROUNDS = 10


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    magpie.build()
    magpie.lib()


def member(m, levels=3, seed=11):
    n, m, g, s, j, B = SIDES[m]
    return Member((n, m, g, s, j, levels, B), seed)


def dev_idx(values):
    return torch.tensor(list(values), dtype=torch.int32, device="cuda")


def reported(ctx):
    with pytest.raises(magpie.MagpieError) as ei:
        magpie.magpie_window_values(ctx)
    assert ei.value.code == magpie.EINDEX


@pytest.mark.parametrize("m", sorted(SIDES))
def test_steps_of_skipped_windows_change_nothing(m):
    """Single windows and whole minibatches, each behind a valid step."""
    mb = member(m)
    ctx = mb.ctx()
    z = mb.zt
    plain = mb.ctx()
    z_plain = mb.zt
    for r in range(ROUNDS):
        good = dev_idx((r + 3 * i) % mb.N for i in range(min(mb.B, 3)))
        bad = dev_idx([mb.N + r] if r % 2 else [mb.N, -1, mb.N + 7, -(1 << 31), (1 << 31) - 1][: mb.B])
        magpie.magpie_step(ctx, good)
        magpie.magpie_step(ctx, bad)
        magpie.magpie_step(plain, good)
        assert torch.equal(z, z_plain)
        reported(ctx)
    ctx.close()
    plain.close()


@pytest.mark.parametrize("m", sorted(SIDES))
def test_sweep_with_a_minibatch_of_skipped_windows(m):
    """A sweep's own permutation with one minibatch out of range: the sweep of
    the others, on a first (launched) and on a later (replayed) sweep."""
    mb = member(m)
    ctx = mb.ctx()
    z = mb.zt
    plain = mb.ctx()
    z_plain = mb.zt
    for sweep in range(4):
        o = orders([mb], sweep)[0]
        at = sweep % -(-mb.N // mb.B) * mb.B
        bad = o.clone()
        bad[at:at + mb.B] = mb.N
        magpie.magpie_sweep(ctx, bad)
        for s in range(0, mb.N, mb.B):
            if s != at:
                magpie.magpie_step(plain, o[s:s + mb.B].contiguous())
        assert torch.equal(z, z_plain)
        reported(ctx)
    ctx.close()
    plain.close()


def test_group_sweep_of_skipped_windows_changes_nothing():
    """Members of one side alone in their launches, and of several sides."""
    members = [member(64), member(128, seed=12), member(128, levels=2, seed=13)]
    ctxs, objects = [], []
    for mb in members:
        ctxs.append(mb.ctx())
        objects.append(mb.zt)
    group = magpie.magpie_group_create(ctxs)
    magpie.magpie_group_set_persistent(group, 0)
    for sweep in range(ROUNDS):
        magpie.magpie_group_sweep(group, orders(members, sweep))
        torch.cuda.synchronize()
        before = [z.clone() for z in objects]
        magpie.magpie_group_sweep(group, [torch.full_like(o, mb.N) for mb, o in zip(members, orders(members, 0))])
        for a, b in zip(before, objects):
            assert torch.equal(a, b)
        for c in ctxs:
            reported(c)
    group.close()
    for c in ctxs:
        c.close()


@pytest.mark.parametrize("path", [1, 2])
@pytest.mark.parametrize("m,levels", [(64, 3), (64, 6), (128, 7)])
def test_precision_steps_with_skipped_windows(m, levels, path):
    """Tensor-core steps hand windows from kernel to kernel by counts that the
    update clears: skipped windows, some or all of a step's, leave the counts and
    the object as a step without them does (the V-cycle inside the gradient
    kernel, and the coarse kernel of deeper cycles)."""
    mb = member(m, levels)
    ctx = mb.ctx()
    z = mb.zt
    plain = mb.ctx()
    z_plain = mb.zt
    for c in (ctx, plain):
        magpie.magpie_set_precision(c, path)
    for r in range(ROUNDS):
        k = r % mb.N
        magpie.magpie_step(ctx, dev_idx([mb.N, k, -1, (k + 2) % mb.N]))
        magpie.magpie_step(ctx, dev_idx([mb.N + r] if r % 2 else [-1, mb.N, mb.N + 3]))
        magpie.magpie_step(plain, dev_idx([k, (k + 2) % mb.N]))
        assert torch.equal(z, z_plain)
        reported(ctx)
    ctx.close()
    plain.close()
