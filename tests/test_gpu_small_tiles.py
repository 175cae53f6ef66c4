"""Launches of few tiles run 32 x 12 tiles: the fields of a pair alone (small tiles at every
level) are, bit for bit, those of the same pair in a batch whose level-0 launches have
enough tiles for the 64-wide ones."""
import pytest

from paper_1306_2461_gb300 import synth
from helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage,H,W", [("f16", 150, 200), ("f32", 97, 129), ("bf16", 121, 321)])
@pytest.mark.parametrize("r,variant", [(r, False) for r in (2, 3, 4, 5, 6, 8, 10)] + [(r, True) for r in (2, 5, 10, 16)])
def test_small_tiles_equal_wide_tiles(storage, H, W, r, variant):
    import torch
    from paper_1306_2461_gb300 import of
    p = synth.make_c1(H, W, seed=H + r)
    I1, I2 = to_dev(p.I1), to_dev(p.I2)
    plan = of.Plan.make(H, W, 2, r, 3, bits=8, storage=storage, flags=of.OF_FLAG_I1GRAD if variant else 0)
    tiles = -(-W // 64) * -(-H // 24)
    n = 4 * torch.cuda.get_device_properties(0).multi_processor_count // (3 * tiles) + 2
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
