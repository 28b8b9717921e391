"""A group whose members of one window side run in different forms (GPU): windows
of 64 in the cluster kernel (minibatches of 65 to 152 windows) beside windows of
64 in the split form, in one update launch, with a second side concurrent.
Every member gets the bits, and the window values, of its own sweeps."""
import pytest
import torch

from paper_2504_10118_gb300 import magpie
from tests.test_gpu_group import Member, orders

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    magpie.build()
    magpie.lib()


# (n, m, grid, step, jitter, levels, minibatch): the cluster form ends first, last and not at all
GROUPS = [[(150, 64, 12, 7, 2, 3, 70), (131, 64, 7, 10, 2, 3, 16), (201, 128, 5, 14, 3, 3, 8)],
          [(131, 64, 4, 17, 2, 4, 6), (180, 64, 18, 6, 1, 2, 152), (150, 64, 12, 7, 2, 5, 144)],
          [(150, 64, 12, 7, 2, 3, 64), (155, 64, 13, 7, 1, 3, 153)]]


@pytest.mark.parametrize("specs", GROUPS)
@pytest.mark.parametrize("shape", [0, 2])
def test_mixed_forms_of_one_side(specs, shape):
    members = [Member(s, 31 + i) for i, s in enumerate(specs)]
    alone, own, grouped, objects = [], [], [], []
    for mb in members:
        alone.append(mb.ctx())
        own.append(mb.zt)
        grouped.append(mb.ctx())
        objects.append(mb.zt)
    group = magpie.magpie_group_create(grouped)
    magpie.magpie_group_set_persistent(group, 0)
    magpie.magpie_group_set_apply_shape(group, shape)
    for sweep in range(3):
        o = orders(members, sweep)
        magpie.magpie_group_sweep(group, o)
        for c, order in zip(alone, o):
            magpie.magpie_sweep(c, order)
        torch.cuda.synchronize()
        for z, want in zip(objects, own):
            assert torch.equal(z, want)
    for c, g in zip(alone, grouped):
        for want, got in zip(magpie.magpie_window_values(c), magpie.magpie_window_values(g)):
            assert torch.equal(want, got)
    group.close()
    for c in alone + grouped:
        c.close()
