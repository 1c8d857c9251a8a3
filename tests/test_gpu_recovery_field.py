"""Primitive recovery in gas that the magnetic field dominates, up to B^2 = 1e9 rho h: the slope of
the master function is a difference of large terms there unless it is formed as a sum of positive
ones.  On a flat Cartesian metric, against the primitives that the state was made of."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import paper_2508_18221_gb300 as pkg                      # noqa: E402

from test_gpu_recovery_cold import LD, U_RND, _state      # noqa: E402


@pytest.mark.parametrize("sigma", [1e2, 1e4, 1e6, 1e7, 1e9])
@pytest.mark.parametrize("w,eps", [(1.001, 1.0), (1.5, 1.0), (5.0, 1.0), (5.0, 100.0), (30.0, 10.0), (300.0, 100.0)])
def test_recovery_returns_the_primitives(w, eps, sigma):
    cfg, U, rho, v, e, W, h = _state(w, eps, sigma, 4.0 / 3.0)
    ctx = pkg.Context(*pkg.make_structs(cfg))
    ctx.set_state(torch.from_numpy(U.reshape(-1).copy()).cuda(), True)
    out = torch.empty(pkg.NPRIM * ctx.n_points, dtype=torch.float64, device="cuda")
    # the roundings of the map (test_gpu_recovery_cold.py) with the field's share of the energy
    unit = 32 * U_RND * (1 + sigma)
    near_floor = int((e <= 2 * unit * h * W ** 2).sum())
    for start in ("reset", "warm"):
        failed = ctx.con2prim(out, True)
        got = out.cpu().numpy().reshape((pkg.NPRIM,) + W.shape).astype(LD)
        assert failed <= near_floor, start
        assert float((np.abs(got[6] / W - 1) / W ** 2).max()) <= unit, start
        assert float((np.abs(got[0] / rho - 1) / W ** 2).max()) <= unit, start
        assert float((np.abs(got[4] - e) / (h * W ** 2)).max()) <= unit, start
        assert float(np.abs(got[1:4] - v).max()) <= unit, start
    ctx.close()
