"""Strips of four tiles (the planes as rings, the estimate and window of a tile requested
while the tile above finishes): a batch with enough tiles for them gives the fields of the
pair alone, bit for bit, at every radius that has strips, staged and gathered, also with the
first image's gradient."""
import pytest

from paper_1306_2461_gb300 import synth
from helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gather", [False, True])
@pytest.mark.parametrize("r,variant", [(r, False) for r in range(2, 13)] + [(r, True) for r in (2, 3, 4, 5, 10, 12)])
def test_strips_equal_single_tiles(r, variant, gather):
    import torch
    from paper_1306_2461_gb300 import of
    H, W = 721 + r, 1003 - r   # ragged: last tile rows of a strip below the image, odd widths
    p = synth.make_c1(H, W, seed=r)
    I1, I2 = to_dev(p.I1), to_dev(p.I2)
    storage = ("f32", "f16", "bf16")[r % 3]
    flags = (of.OF_FLAG_GATHER if gather else 0) | (of.OF_FLAG_I1GRAD if variant else 0)
    plan = of.Plan.make(H, W, 2, r, 3, bits=8, storage=storage, flags=flags)
    # strips of 4 from 8 blocks per SM on
    tiles = -(-W // 64) * -(-H // 24)
    n = 32 * torch.cuda.get_device_properties(0).multi_processor_count // tiles + 1
    with of.Flow(plan) as f:
        u, v = f.compute(I1, I2)
        torch.cuda.synchronize()
        assert f.sync_status() == of.OF_OK
    flows = [of.Flow(plan) for _ in range(n)]
    us, vs = of.compute_batch(flows, [I1] * n, [I2] * n)
    torch.cuda.synchronize()
    for f, ub, vb in zip(flows, us, vs):
        assert f.sync_status() == of.OF_OK
        assert torch.equal(u, ub) and torch.equal(v, vb)
        f.close()
