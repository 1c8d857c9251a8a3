"""A line that holds an Inf or a NaN has NaN derivatives, whatever the size of the operator's
entries (radial coordinates in units that make them tiny)."""
import numpy as np
import pytest

from workloads import config

from test_gpu_parity import _ctx, pkg  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r_max", [20.0, 1e12, 1e25])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_radial_lines(pkg, r_max, bad):  # noqa: F811
    torch = pytest.importorskip("torch")
    cfg = config("c1", n_elem=1, n_r=24, n_theta=12, n_phi=16, r_min=0.1 * r_max, r_max=r_max)
    ctx = _ctx(pkg, cfg)
    u = np.random.default_rng(2).standard_normal((1, 24, 12, 16))
    u[0, 5, 3, 7] = bad
    src = torch.from_numpy(u).cuda()
    dst = torch.empty_like(src)
    ctx.debug_deriv(src, dst, 1, 0)
    got = dst.cpu().numpy()[0]
    line = np.zeros((12, 16), dtype=bool)
    line[3, 7] = True
    assert np.isnan(got[:, line]).all()
    assert np.isfinite(got[:, ~line]).all()
    ctx.close()
