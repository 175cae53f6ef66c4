"""Gathered phase launches of the radii that have a kernel of their own for them: every strip
length, with the L2 prefetch and in two sequences, gives the pair's fields bit for bit."""
import pytest

from paper_1306_2461_gb300 import synth
from helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r,storage", [(5, "f16"), (6, "f32")])
def test_gathered_batch_equals_the_pair(r, storage):
    import torch
    from paper_1306_2461_gb300 import of
    H, W = 721 + r, 1003 - r
    p = synth.make_c1(H, W, seed=r)
    I1, I2 = to_dev(p.I1), to_dev(p.I2)
    plan = of.Plan.make(H, W, 2, r, 3, bits=8, storage=storage)
    with of.Flow(plan) as f:
        u, v = f.compute(I1, I2)
        torch.cuda.synchronize()
    # level-0 tiles for strips of 4: four times two blocks on each of an SM's three slots
    n = 24 * torch.cuda.get_device_properties(0).multi_processor_count // (-(-W // 64) * -(-H // 24)) + 1
    assert n <= 64   # pairs of one launch
    flows = [of.Flow(plan) for _ in range(n)]
    sc, s = of.batch_size_class(flows), torch.cuda.Stream()
    for t in ({}, {"strip": 2}, {"strip": 1}, {"prefetch": 1}, {"branches": 2}):
        of.tuning_set(plan, sc, stage_i2=0, **t)
        us, vs = of.compute_batch(flows, [I1] * n, [I2] * n, stream=s)
        torch.cuda.synchronize()
        for f, ub, vb in zip(flows, us, vs):
            assert f.sync_status() == of.OF_OK
            assert torch.equal(u, ub) and torch.equal(v, vb), t
    of.tuning_clear()
    for f in flows:
        f.close()
