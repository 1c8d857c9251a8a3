"""Primitive recovery at the ends of its range, against the oracle's bisection: slow and fast
flows, cold and hot gas, weak and strong fields, node counts that end inside a block."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import paper_2508_18221_gb300 as pkg                      # noqa: E402
from oracle import solver as so                           # noqa: E402
from oracle import valencia as va                         # noqa: E402
from workloads import config                              # noqa: E402

U_RND = 2.0 ** -53


@pytest.mark.parametrize("warm", [False, True])
@pytest.mark.parametrize("shape,w_max,eps,beta_inv", [
    ((1, 4, 4, 4), 1.0 + 1e-9, 1e-6, 0.0),        # nearly at rest, cold, no field
    ((1, 7, 5, 6), 1.2, 1e-3, 1e-2),
    ((2, 9, 11, 6), 10.0, 1.0, 1.0),
    ((1, 5, 13, 10), 50.0, 1e2, 10.0),            # fast, hot, strongly magnetised
    ((1, 6, 6, 8), 5.0, 1e-5, 1e3),               # cold, dominated by the field
])
def test_recovery_extremes(shape, w_max, eps, beta_inv, warm):
    cfg = config("c1", n_elem=shape[0], n_r=shape[1], n_theta=shape[2], n_phi=shape[3])
    g, p, U = so.workload_state(cfg)
    gam, sqg = so.metric_from_bssn(so.unpack_bssn(U))
    rng = np.random.default_rng(7)
    n = g.shape
    # a direction and a Lorentz factor between 1 and w_max; field of random direction
    L = np.linalg.cholesky(gam)
    unit = lambda: (lambda x: x / np.linalg.norm(x, axis=-1, keepdims=True))(rng.standard_normal(n + (3,)))
    up = lambda x: np.linalg.solve(np.swapaxes(L, -1, -2), x[..., None])[..., 0]
    W = 1.0 + (w_max - 1.0) * rng.random(n)
    v = up(unit()) * np.sqrt(1.0 - 1.0 / W ** 2)[..., None]
    rho = 10.0 ** rng.uniform(-6, 0, n)
    e = eps * (1.0 + rng.random(n))
    pr = (p.gamma_eos - 1.0) * rho * e
    B = up(unit()) * np.sqrt(2.0 * beta_inv * pr)[..., None]
    D, S, tau, _ = va.prim_to_cons(rho, v, e, B, U[so.I_ALPHA], np.moveaxis(U[so.I_BETA:so.I_BETA + 3], 0, -1), gam,
                                   p.gamma_eos)
    U[so.I_D], U[so.I_TAU] = sqg * D, sqg * tau
    for i in range(3):
        U[so.I_S + i], U[so.I_B + i] = sqg * S[..., i], sqg * B[..., i]
    ref = so.primitives(U, p)
    ctx = pkg.Context(*pkg.make_structs(cfg))
    Ud = torch.from_numpy(U.reshape(-1).copy()).cuda()
    ctx.set_state(Ud, True)
    out = torch.empty(pkg.NPRIM * ctx.n_points, dtype=torch.float64, device="cuda")
    nf = ctx.con2prim(out, True)
    if warm:
        nf = ctx.con2prim(out, True)
    got = out.cpu().numpy().reshape((pkg.NPRIM,) + n)
    ctx.close()
    # Both solve the same equations from the same rounded inputs, so they differ by the
    # rounding of the map: eps is a difference of terms of size s = h W^2 (1 + B^2 / (rho h))
    # (energy per rest mass), a few tens of roundings of it on either side; W, rho and v move
    # with the momentum, whose relative rounding W^2 multiplies.
    s = (1.0 + p.gamma_eos * e + 2.0 * beta_inv * pr / rho) * W ** 2
    tol_e = 100.0 * U_RND * s * W ** 2
    assert np.all(np.abs(got[4] - ref["eps"]) <= tol_e + 1e-13 * ref["eps"])
    rel = 100.0 * U_RND * s * W ** 2
    assert np.all(np.abs(got[6] / ref["W"] - 1.0) <= rel)
    assert np.all(np.abs(got[0] / ref["rho"] - 1.0) <= rel)
    for i in range(3):
        assert np.all(np.abs(got[1 + i] - ref["v"][..., i]) <= rel * np.abs(up(np.ones(n + (3,)))).max())
    # counted points: the same but for values within their rounding of the floor
    near = np.sum(np.abs(ref["eps"] - p.eps_atm) <= tol_e)
    assert abs(nf - int(np.sum(~ref["ok"]))) <= near
