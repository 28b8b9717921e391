"""A step on an object much larger than its windows (GPU): what the windows do
not touch is neither changed nor read."""
import numpy as np
import pytest
import torch

from paper_2504_10118_gb300 import magpie, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    magpie.build()
    magpie.lib()


def context(n, m, B, precision=0):
    dev = torch.device("cuda")
    rng = np.random.default_rng(m)
    pos = rng.integers(0, n - m + 1, (B, 2)).astype(np.int32)
    z = torch.ones((n, n), dtype=torch.complex64, device=dev)
    Q = torch.from_numpy(synth.make_probe(m).astype(np.complex64)).to(dev)
    post = torch.from_numpy(pos).to(dev)
    d = 1.5 * magpie.magpie_forward_intensities(z, Q, post, m)
    ctx = magpie.magpie_create(magpie.magpie_params_of(n, n, m, B, 2, B, 0.5), z, Q, post, d)
    if precision:
        magpie.magpie_set_precision(ctx, precision)
    return ctx, z, pos


def least_us(call, calls=10, rounds=5):
    best = float("inf")
    for _ in range(rounds):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(calls):
            call()
        b.record()
        torch.cuda.synchronize()
        best = min(best, 1e3 * a.elapsed_time(b) / calls)
    return best


@pytest.mark.parametrize("m,precision", [(32, 0), (64, 0), (128, 1)])
def test_step_leaves_the_rest_of_a_large_object_alone(m, precision):
    """Eight windows on 16384 x 16384 pixels (2 GiB).  A step that skips the tiles
    without windows is bound by the launch of a block per 32 x 32 tile, 1.0 to
    1.1 times what one read of the object takes (half of a copy of it, timed
    here); with the tiles read as well it took 1.8 times: the line lies between."""
    n, B = 16384, 8
    ctx, z, pos = context(n, m, B, precision)
    idx = torch.arange(B, dtype=torch.int32, device="cuda")
    magpie.magpie_step(ctx, idx)
    torch.cuda.synchronize()
    inside = torch.zeros((n, n), dtype=torch.bool, device="cuda")
    for r, c in pos:
        inside[r:r + m, c:c + m] = True
    changed = z != 1
    assert bool((changed & inside).any()) and not bool((changed & ~inside).any())
    del inside, changed
    copy = torch.empty_like(z)
    read = least_us(lambda: copy.copy_(z)) / 2
    del copy
    step = least_us(lambda: magpie.magpie_step(ctx, idx))
    print(f"m {m}: step {step:.0f} us, a read of the object {read:.0f} us")
    assert step < 1.4 * read
    ctx.close()
