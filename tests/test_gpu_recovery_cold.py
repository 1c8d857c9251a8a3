"""Primitive recovery where 1 - v^2 and the specific energy lie below what FP32 resolves: cold
gas at any speed, hot gas up to W = 1e4.  On a flat Cartesian metric the recovery alone rounds,
and the exact primitives are those that the conserved state was made of."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import paper_2508_18221_gb300 as pkg                      # noqa: E402
from oracle import solver as so                           # noqa: E402
from workloads import config                              # noqa: E402

U_RND = 2.0 ** -53
LD = np.longdouble


def _state(w, eps, sigma, gamma):
    """Conserved state of gas with W in [1 + 0.8 (w - 1), w], energies in [eps, 2 eps] and field
    energy B^2 = sigma rho h, and its primitives."""
    cfg = config("c1")
    g, _, U = so.workload_state(cfg)
    n = g.shape
    U = np.zeros_like(U)
    U[0], U[3], U[5], U[so.I_ALPHA] = 1.0, 1.0, 1.0, 1.0
    rng = np.random.default_rng(3)
    unit = lambda: (lambda x: x / np.sqrt((x * x).sum(axis=0)))(rng.standard_normal((3,) + n).astype(LD))  # noqa: E731
    W = (1 + (w - 1) * (0.8 + 0.2 * rng.random(n))).astype(LD)
    rho = (10.0 ** rng.uniform(-6, 0, n)).astype(LD)
    e = (eps * (1 + rng.random(n))).astype(LD)
    p = (LD(gamma) - 1) * rho * e
    h = 1 + LD(gamma) * e
    v = unit() * np.sqrt(1 - 1 / W ** 2)
    B = (unit() * np.sqrt(sigma * rho * h)).astype(np.float64).astype(LD)
    Z, B2, vB = rho * h * W ** 2, (B * B).sum(axis=0), (v * B).sum(axis=0)
    U[so.I_D] = rho * W
    U[so.I_S:so.I_S + 3] = (Z + B2) * v - vB * B
    U[so.I_TAU] = Z + B2 - p - (B2 / W ** 2 + vB ** 2) / 2 - rho * W
    U[so.I_B:so.I_B + 3] = B
    return cfg, U, rho, v, e, W, h


@pytest.mark.parametrize("sigma", [0.0, 1.0])
@pytest.mark.parametrize("w,eps", [
    (1.01, 1e-8), (1.5, 1e-8), (5.0, 1e-9), (5.0, 1e-7), (5.0, 1e-4), (10.0, 1e-9), (10.0, 1e-6),
    (30.0, 1e-8), (30.0, 1e-6), (100.0, 1e-9), (100.0, 1e-8), (100.0, 1e-4),      # cold
    (300.0, 1e-8), (1000.0, 1e-4), (1000.0, 1.0), (3000.0, 1e2), (10000.0, 1.0),  # beyond FP32's 1 - v^2
])
def test_recovery_returns_the_primitives(w, eps, sigma):
    cfg, U, rho, v, e, W, h = _state(w, eps, sigma, 4.0 / 3.0)
    grid, phys, opts = pkg.make_structs(cfg)
    assert phys.gamma_eos == 4.0 / 3.0 and phys.eps_atm <= 1e-10
    ctx = pkg.Context(grid, phys, opts)
    ctx.set_state(torch.from_numpy(U.reshape(-1).copy()).cuda(), True)
    out = torch.empty(pkg.NPRIM * ctx.n_points, dtype=torch.float64, device="cuda")
    # v^2 takes some sixteen roundings (of S^2 / D^2, of the root mu, of their product); they move W
    # by W^2 / 2 of that and eps by h W^2, relative to the energy per rest mass with the field's
    # share; twice that for the rounding of the inputs: 32 units
    unit = 32 * U_RND * (1 + sigma)
    for start in ("reset", "warm"):
        failed = ctx.con2prim(out, True)
        got = out.cpu().numpy().reshape((pkg.NPRIM,) + W.shape).astype(LD)
        assert failed == 0, start
        assert float((np.abs(got[6] / W - 1) / W ** 2).max()) <= unit, start
        assert float((np.abs(got[0] / rho - 1) / W ** 2).max()) <= unit, start
        assert float((np.abs(got[4] - e) / (h * W ** 2)).max()) <= unit, start
        assert float(np.abs(got[1:4] - v).max()) <= unit, start
    ctx.close()


def test_iteration_limit():
    """c2p_maxit = 1: one FP64 step does not bring the search's FP32 root to c2p_tol, so every
    node counts as failed; the default solves all of them."""
    cfg, U, *_ = _state(5.0, 1e-3, 0.0, 4.0 / 3.0)
    state = torch.from_numpy(U.reshape(-1).copy()).cuda()
    for maxit in (1, None):
        ctx = pkg.Context(*pkg.make_structs(cfg, **({} if maxit is None else {"c2p_maxit": maxit})))
        ctx.set_state(state, True)
        out = torch.empty(pkg.NPRIM * ctx.n_points, dtype=torch.float64, device="cuda")
        assert ctx.con2prim(out, True) == (0 if maxit is None else ctx.n_points)
        ctx.close()
