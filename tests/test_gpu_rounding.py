"""The fixed-radius kernels round no more than the run-time-radius kernel, which refers the FP32
right-hand side of each 64 x 24 tile (64 x 32 in the variant) to the estimate at its centre: the
error against FP64 of the radii and the variant that ran that kernel before they had their own."""
import numpy as np
import pytest

from paper_1306_2461_gb300 import synth
from helpers import oracle_flow_stored, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r,variant", [(7, False), (12, False), (13, False), (16, False), (4, True), (10, True)])
def test_error_of_the_fixed_radius_kernels(oracle_mod, r, variant):
    # 95th percentile away from the border; the window sums of a group share additions, so their
    # order is another one: a quarter more is allowed for that (a reference four tiles away doubles it)
    import torch
    from paper_1306_2461_gb300 import of
    H, W, L, n = 300, 700, 3, 3
    p = synth.make_c2(H, W, seed=r)
    uo, vo = oracle_flow_stored(oracle_mod, p.I1, p.I2, L, r, n, "f32", i1grad=variant)
    I1, I2 = to_dev(p.I1), to_dev(p.I2)
    plan = of.Plan.make(H, W, L, r, n, bits=12, storage="f32", flags=of.OF_FLAG_I1GRAD if variant else 0)
    m, err = 4 * (r + 2), []
    with of.Flow(plan) as f:
        sc = of.batch_size_class([f])
        for generic in (1, 0):
            of.tuning_set(plan, sc, generic_sums=generic, stage_i2=1 - generic, strip=1 if generic else 4)
            us, vs = of.compute_batch([f], [I1], [I2])
            torch.cuda.synchronize()
            assert f.sync_status() == of.OF_OK
            d = np.maximum(np.abs(us[0].cpu().double().numpy() - uo), np.abs(vs[0].cpu().double().numpy() - vo))
            err.append(float(np.quantile(d[m:-m, m:-m], 0.95)))
        of.tuning_clear()
    print(f"r={r} variant={variant}: 95th percentile {err[0]:.3e} run-time radius, {err[1]:.3e} fixed")
    assert err[1] <= 1.25 * err[0]
