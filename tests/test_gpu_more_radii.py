"""Window radii with the per-pair and phase kernels only: fields against the oracle on every
pixel, and the same bits alone (small tiles), gathered, and in a batch (wide tiles, in
strips where the radius allows them)."""
import numpy as np
import pytest

from paper_1306_2461_gb300 import synth
from helpers import gpu_flow, parity_check, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,storage", [(97, 129, "f32"), (150, 70, "f16")])
@pytest.mark.parametrize("r", [7, 9, 11, 12, 13, 14, 15, 16])
def test_radius_matches_oracle_and_batch(oracle_mod, r, H, W, storage):
    import torch
    from paper_1306_2461_gb300 import of
    I1, I2 = synth.translated_texture_pair(H, W, (0.7, -0.4), seed=r + H, amp=800.0, offset=2000.0, fmax=1.0 / 8.0)
    I1, I2 = np.rint(I1).astype(np.uint16), np.rint(I2).astype(np.uint16)
    u, v = gpu_flow((I1, I2), 2, r, 2, storage, bits=12)
    parity_check(u, v, (I1, I2), oracle_mod, 2, r, 2, storage, f"r={r} {H}x{W}", margin=0, workload=False)
    ug, vg = gpu_flow((I1, I2), 2, r, 2, storage, bits=12, flags=of.OF_FLAG_GATHER)
    assert np.array_equal(u, ug) and np.array_equal(v, vg)
    plan = of.Plan.make(H, W, 2, r, 2, bits=12, storage=storage)
    n = 60   # more 64 x 24 tiles than 16 blocks per SM at level 0: strips of 2
    n = max(n, 16 * torch.cuda.get_device_properties(0).multi_processor_count // (-(-W // 64) * -(-H // 24)) + 1)
    flows = [of.Flow(plan) for _ in range(n)]
    us, vs = of.compute_batch(flows, [to_dev(I1)] * n, [to_dev(I2)] * n)
    torch.cuda.synchronize()
    for k, f in enumerate(flows):
        assert f.sync_status() == of.OF_OK
        f.close()
    for k in (0, n // 2, n - 1):
        assert np.array_equal(us[k].cpu().double().numpy(), u) and np.array_equal(vs[k].cpu().double().numpy(), v)


@pytest.mark.parametrize("r", [7, 12, 16])
def test_variant_at_these_radii(oracle_mod, r):
    from paper_1306_2461_gb300 import of
    I1, I2 = synth.translated_texture_pair(70, 100, (0.6, 0.5), seed=r, amp=800.0, offset=2000.0, fmax=1.0 / 8.0)
    I1, I2 = np.rint(I1).astype(np.uint16), np.rint(I2).astype(np.uint16)
    u, v = gpu_flow((I1, I2), 2, r, 2, "f32", bits=12, flags=of.OF_FLAG_I1GRAD)
    parity_check(u, v, (I1, I2), oracle_mod, 2, r, 2, "f32", f"variant r={r}", margin=0, workload=False, i1grad=True)


@pytest.mark.parametrize("r", [7, 16])
def test_tunings_of_forms_these_radii_lack(r):
    # accepted as before, and run as the phase launches or with per-output sums
    import torch
    from paper_1306_2461_gb300 import of
    p = synth.make_c1(100, 130, seed=r)
    I1, I2 = to_dev(p.I1), to_dev(p.I2)
    plan = of.Plan.make(100, 130, 2, r, 3, bits=8)
    res = []
    with of.Flow(plan) as f:
        sc = of.batch_size_class([f])
        for t in ({}, {"tile_h": 32}, {"phased": 0, "blocks_per_sm": 2, "stage_i2": 0, "strip": 1},
                  {"generic_sums": 1, "stage_i2": 0, "strip": 1}):
            of.tuning_set(plan, sc, **t)
            us, vs = of.compute_batch([f], [I1], [I2])
            torch.cuda.synchronize()
            assert f.sync_status() == of.OF_OK
            res.append((us[0].clone(), vs[0].clone()))
        of.tuning_clear()
        with pytest.raises(of.OfError):
            of.tuning_set(plan, sc, fusion=2)
        best, cands = of.autotune_batch([f], [I1], [I2], reps=1)
        of.tuning_clear()
    assert any(c["generic_sums"] == 0 for c in cands) and all(c["tile_h"] == 24 for c in cands)
    for u, v in res[1:3]:
        assert torch.equal(u, res[0][0]) and torch.equal(v, res[0][1])
