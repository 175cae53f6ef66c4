"""The forms a batch runs by default on a stream of the caller's (a replayed graph, two launch
sequences, strips of each length, small tiles), with an L2 prefetch, and a pair captured by the
caller, against the pair alone on the default stream (chained launches), bit for bit."""
import pytest

from paper_1306_2461_gb300 import synth
from helpers import to_dev

pytestmark = pytest.mark.gpu


def pair(H, W, r, L, variant, storage):
    import torch
    from paper_1306_2461_gb300 import of
    p = synth.make_c1(H, W, seed=H + r)
    I1, I2 = to_dev(p.I1), to_dev(p.I2)
    plan = of.Plan.make(H, W, L, r, 3, bits=8, storage=storage, flags=of.OF_FLAG_I1GRAD if variant else 0)
    with of.Flow(plan) as f:
        u, v = f.compute(I1, I2)
        torch.cuda.synchronize()
        assert f.sync_status() == of.OF_OK
    return plan, I1, I2, u, v


RADII = [(r, False) for r in range(2, 17)] + [(r, True) for r in (2, 4, 7, 10, 16)]


@pytest.mark.parametrize("r,variant", RADII)
def test_batch_on_a_stream_equals_the_pair(r, variant):
    # two sequences of n/2 pairs, each with the level-0 tiles for strips of 4 (four times the resident
    # slots, of which an SM has at most four), 45 rows of tiles (a remainder in each column's last
    # strip), shorter strips at level 1 and small tiles at the coarsest
    import torch
    from paper_1306_2461_gb300 import of
    H, W = 1061 + r, 835 - r
    plan, I1, I2, u, v = pair(H, W, r, 4, variant, ("f32", "f16", "bf16")[r % 3])
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    tiles = -(-W // 64) * -(-H // 24)
    n = 2 * (16 * sms // tiles + 1)   # at most four slots per SM
    assert n // 2 * tiles >= 4 * 4 * sms and n // 2 <= 64
    flows, s = [of.Flow(plan) for _ in range(n)], torch.cuda.Stream()
    for t in (None, {"prefetch": 1}, {"prefetch": 2, "branches": 2, "strip": 2}):
        if t is not None:
            of.tuning_set(plan, of.batch_size_class(flows), **t)
        us, vs = [torch.zeros_like(u) for _ in range(n)], [torch.zeros_like(v) for _ in range(n)]
        torch.cuda.synchronize()
        for _ in range(2):   # captured, then replayed
            of.compute_batch(flows, [I1] * n, [I2] * n, us, vs, stream=s)
        s.synchronize()
        for f, a, b in zip(flows, us, vs):
            assert f.sync_status() == of.OF_OK
            assert torch.equal(u, a) and torch.equal(v, b), t
    of.tuning_clear()
    for f in flows:
        f.close()


@pytest.mark.parametrize("H,W", [(150, 200), (700, 900)])
@pytest.mark.parametrize("r,variant", [(4, False), (9, False), (16, False), (5, True)])
def test_pair_in_a_callers_capture(H, W, r, variant):
    import torch
    from paper_1306_2461_gb300 import of
    plan, I1, I2, u, v = pair(H, W, r, 3, variant, "f32")
    a, b = torch.zeros_like(u), torch.zeros_like(v)
    with of.Flow(plan) as f:
        g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        torch.cuda.synchronize()
        with torch.cuda.graph(g, stream=s):
            f.compute(I1, I2, a, b, stream=s)
        for _ in range(2):
            a.zero_(), b.zero_()
            g.replay()
            torch.cuda.synchronize()
            assert torch.equal(u, a) and torch.equal(v, b)
        f.compute(I1, I2, a, b)   # the handle is released after work outside a capture
        torch.cuda.synchronize()
        assert torch.equal(u, a) and torch.equal(v, b)
