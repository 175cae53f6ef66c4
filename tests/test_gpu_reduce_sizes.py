"""The reductions of a field at the sizes where their forms change: one value, tails of the
16-byte loads, fields that start off a 16-byte boundary, either side of the largest field one
cluster takes, and infinities, NaN and signed zeros."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W", [(1, 1), (1, 5), (3, 1027), (1024, 1024), (1, (1 << 20) + 1), (1531, 1201)])
@pytest.mark.parametrize("offset", [0, 1])
def test_count_and_extremes(H, W, offset):
    import torch
    from paper_1306_2461_gb300 import of
    rng = np.random.default_rng(H + W)
    a = rng.normal(0.0, 2.0, H * W).astype(np.float32)
    a[::11] = np.nan
    a[::17] = -0.0
    buf = torch.empty(H * W + 1, device="cuda")
    u = buf[offset:offset + H * W].view(H, W)
    u.copy_(torch.from_numpy(a).view(H, W))
    for Tv in (-0.5, 0.0, np.inf):
        assert int(of.sbubble(u, Tv)) == int((a <= np.float32(Tv)).sum())
    lo, hi = of.field_minmax(u).cpu().numpy()
    if np.isnan(a).all():
        assert np.isnan(lo) and np.isnan(hi)
    else:
        assert lo == np.nanmin(a) and hi == np.nanmax(a)
    u[-1, -1] = np.inf
    u[0, 0] = -np.inf if H * W > 1 else np.inf
    lo, hi = of.field_minmax(u).cpu().numpy()
    assert hi == np.inf and lo == (-np.inf if H * W > 1 else np.inf)


def test_zero_signs():
    import torch
    from paper_1306_2461_gb300 import of
    z = torch.zeros(4, 300, device="cuda")
    z[2, 7] = -0.0
    lo, hi = of.field_minmax(z).cpu().numpy()
    assert np.signbit(lo) and not np.signbit(hi)
