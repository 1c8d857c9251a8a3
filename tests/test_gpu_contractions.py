"""The FP64-unit and the mixed-precision contractions at the edges of their tiles: the
smallest and largest sizes, odd ones, and those around the sizes where the kernels change
their warps per block."""
import math

import numpy as np
import pytest

from oracle import solver as so
from oracle import rounding as fpf
from workloads import config

from test_gpu_parity import _ctx, _gpu_rhs, _oracle, assert_parity, pkg  # noqa: F401

pytestmark = pytest.mark.gpu

U_RND = 2.0 ** -53


def _matrix(direction, n, scale):
    """Differentiation matrix in extended precision: barycentric form on the Chebyshev nodes,
    closed form on the Fourier nodes."""
    ld = np.longdouble
    pi = 4 * np.arctan(ld(1))
    if direction == 2:
        d = np.arange(n)
        row = np.zeros(n, dtype=ld)
        row[1:] = ld(0.5) * (-1.0) ** d[1:] / np.tan(pi * d[1:].astype(ld) / n)
        row[n // 2] = 0
        return row[(d[:, None] - d[None, :]) % n]
    i = np.arange(n).astype(ld)
    x = -np.cos(pi * i / (n - 1)) if direction == 0 else -np.cos(pi * (2 * i + 1) / (2 * n))
    dx = x[:, None] - x[None, :]
    np.fill_diagonal(dx, 1)
    w = 1 / np.prod(2 * dx, axis=1)
    m = (w[None, :] / w[:, None]) / dx
    np.fill_diagonal(m, 0)
    np.fill_diagonal(m, -m.sum(axis=1))
    return m * ld(scale)


@pytest.mark.parametrize("shape", [
    (1, 4, 4, 4), (2, 5, 6, 6), (1, 17, 16, 18),      # np = 2 .. 9 pairs: one to four per warp
    (3, 33, 31, 34), (1, 64, 65, 66),                 # odd middle nodes, more than one round of pairs
    (1, 6, 97, 98), (1, 5, 128, 128),                 # the largest
])
def test_fp64_unit_derivatives(pkg, shape):  # noqa: F811
    torch = pytest.importorskip("torch")
    cfg = config("c1", n_elem=shape[0], n_r=shape[1], n_theta=shape[2], n_phi=shape[3])
    ctx = _ctx(pkg, cfg, contraction=1)
    g = so.Grid(so.Params.from_config(cfg))
    u = np.random.default_rng(5).standard_normal((2,) + shape)
    src = torch.from_numpy(u.copy()).cuda()
    dst = torch.empty_like(src)
    for d in range(3):
        ctx.debug_deriv(src, dst, 2, d)
        got = dst.cpu().numpy()
        for e in range(shape[0]):
            n = shape[1 + d]
            scale = (g.r_scale[e], g.t_scale, 1.0)[d]
            D = _matrix(d, n, scale)
            ref = np.moveaxis(np.tensordot(D, u[:, e].astype(np.longdouble), axes=(1, 1 + d)), 0, 1 + d)
            # an n-term dot product (Higham 3.1) with rounded entries: n + 4 roundings of
            # sum |D_ij| max |u|; the nodes' own rounding moves an entry by up to ~n^2 ulp on
            # Chebyshev nodes (spacing ~1/n^2)
            bound = (n + 4 + (n * n if d < 2 else 0)) * U_RND * float(np.abs(D).sum(axis=1).max()) * np.abs(u[:, e]).max()
            assert np.abs(got[:, e] - ref.astype(float)).max() <= bound, (d, n)
    ctx.close()


@pytest.mark.parametrize("shape", [
    (1, 32, 5, 4), (1, 33, 4, 6),                     # the last size of one warp group, the first of two
    (2, 6, 64, 6), (1, 4, 65, 4),                     # of two and of four, along theta
    (1, 5, 6, 66), (1, 4, 4, 128), (2, 7, 9, 30),     # along phi; lines that no 16-byte FP32 load fits
])
def test_mixed_rhs_at_tile_edges(pkg, shape):  # noqa: F811
    cfg = config("c1", n_elem=shape[0], n_r=shape[1], n_theta=shape[2], n_phi=shape[3])
    g, p, U = _oracle(cfg)
    ctx = _ctx(pkg, cfg, precision=1)
    R = _gpu_rhs(pkg, ctx, U)
    ctx.close()
    fn = lambda X: so.rhs(X, g, p)  # noqa: E731
    # the mixed bar (2e-6 of each component's largest value, or its rounding floor at FP32's
    # unit where it is a residue), with the FP64 bar's ten floors: long lines add K roundings
    worst, _ = assert_parity(R, fn(U), f"mixed rhs {shape}", fn, U, tol=2e-6, eps=fpf.EPS32, kappa=10.0)
    assert worst > 1e-12 and math.isfinite(worst)
