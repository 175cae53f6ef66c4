"""A captured batch belongs to its method: closing the handles and opening others of the same
sizes gets the same workspace addresses back, and the new method's batch on the same buffers
and stream must not replay the old one's launches."""
import pytest

from paper_1306_2461_gb300 import synth
from helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("stream", [True, False])
@pytest.mark.parametrize("old,new", [({"storage": "f16"}, {"storage": "bf16"}),
                                     ({"fp64_cond": 1e3}, {"fp64_cond": 0.0})])
def test_batch_of_another_method_on_the_same_buffers(old, new, stream):
    import torch
    from paper_1306_2461_gb300 import of
    H, W, n = 150, 200, 2
    p = synth.make_c1(H, W, seed=5)
    I1, I2 = [to_dev(p.I1)] * n, [to_dev(p.I2)] * n
    plans = [of.Plan.make(H, W, 3, 2, 4, bits=8, **{"storage": "f16", **m}) for m in (old, new)]
    want = []
    for plan in plans:
        with of.Flow(plan) as f:
            want.append([t.clone() for t in f.compute(I1[0], I2[0])])
        torch.cuda.synchronize()
    assert not torch.equal(want[0][0], want[1][0])
    us, vs = ([torch.empty(H, W, device="cuda") for _ in range(n)] for _ in range(2))
    s = torch.cuda.Stream() if stream else None
    for plan, (u, v) in zip(plans, want):
        flows = [of.Flow(plan) for _ in range(n)]
        of.compute_batch(flows, I1, I2, us, vs, stream=s)
        torch.cuda.synchronize()
        for i in range(n):
            assert torch.equal(us[i], u) and torch.equal(vs[i], v)
            flows[i].close()
