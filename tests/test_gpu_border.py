"""Samples near the image border: every pixel of small images whose displacement carries
the sample positions past each side, against the oracle, staged and gathered."""
import numpy as np
import pytest

from paper_1306_2461_gb300 import synth
from helpers import gpu_flow, parity_check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W", [(40, 72), (25, 130), (97, 65)])
@pytest.mark.parametrize("d", [(1.6, 1.2), (-1.6, 1.2), (1.6, -1.2), (-1.6, -1.2)])
def test_border_samples_every_pixel(oracle_mod, H, W, d):
    # one level, so the whole displacement acts at full resolution; a smooth 12-bit texture,
    # compared over every pixel with the FP32 implementation bound (1e-3 px)
    from paper_1306_2461_gb300 import of
    I1, I2 = synth.translated_texture_pair(H, W, d, seed=3 * H + W, amp=800.0, offset=2000.0, fmax=1.0 / 10.0)
    I1, I2 = np.rint(I1).astype(np.uint16), np.rint(I2).astype(np.uint16)
    u, v = gpu_flow((I1, I2), 1, 4, 3, "f32", bits=12)
    parity_check(u, v, (I1, I2), oracle_mod, 1, 4, 3, "f32", f"{H}x{W} {d}", margin=0, workload=False)
    ug, vg = gpu_flow((I1, I2), 1, 4, 3, "f32", bits=12, flags=of.OF_FLAG_GATHER)
    assert np.array_equal(u, ug) and np.array_equal(v, vg)
