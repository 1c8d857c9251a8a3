"""Small grids run their contractions on the integer units (every direction in one launch),
large ones on the tensor cores; both form the same digit sums, so the results are the same
bits.  An instance alone (small) is compared with the same instance inside a batch group
that is too large for the small form."""
import math

import numpy as np
import pytest

from workloads import config

from test_gpu_parity import pkg  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

SPHERE = dict(theta_min=0.0, theta_max=math.pi, theta_basis=1)


@pytest.mark.parametrize("shape,grid,opts", [
    ((2, 12, 12, 16), {}, {}),
    ((3, 9, 11, 6), {}, dict(integrator=1)),                     # odd node counts, RK4
    ((1, 4, 4, 4), {}, dict(filter=63)),                         # smallest; theta filter on every variable
    ((2, 5, 33, 10), {}, dict(glm=1, filter=0)),                 # GLM, no filter, a line of 33 (nine words)
    ((1, 7, 64, 34), {}, dict(filter=34, coupling=1)),           # one direction per group
    ((1, 5, 64, 6), {}, dict(filter=34, coupling=1)),            # longest theta line
    ((2, 64, 5, 8), {}, dict(evolve_metric=0)),                  # longest radial line
    ((2, 6, 8, 64), {}, dict(precision=1)),                      # mixed: the filter alone takes this path
    ((2, 7, 9, 8), SPHERE, dict(filter=63)),                     # Fourier theta: fold inside the kernel
    ((3, 8, 12, 12), SPHERE, dict(glm=1)),
    ((2, 6, 6, 20), SPHERE, dict(precision=1)),
])
def test_small_form_is_bitwise_the_large_form(pkg, shape, grid, opts):  # noqa: F811
    import torch
    from oracle import solver as so
    cfg = config("c1", n_elem=shape[0], n_r=shape[1], n_theta=shape[2], n_phi=shape[3], **grid)
    one = pkg.make_structs(cfg, **opts)
    _, _, U = so.workload_state(cfg, glm=opts.get("glm", 0))
    dt = 1e-6 if grid else 1e-4
    # more nodes x lengths than the small form takes
    n = 3000000 // (U[0].size * sum(shape[1:])) + 1
    batch = pkg.Batch([one] * n)
    state = torch.from_numpy(U.reshape(-1).copy()).cuda()
    for i in range(n):
        batch.set_state(i, state, True)
    batch.step([dt] * n, 2)
    got = np.empty(U.size)
    batch.get_state(n - 1, got, False)
    batch.close()
    # alone, as a batch of one: no check of the state at the end (4 filtered nodes per direction
    # do not carry the black hole; both forms must then give the same NaN)
    alone = pkg.Batch([one])
    alone.set_state(0, state, True)
    alone.step([dt], 2)
    ref = np.empty(U.size)
    alone.get_state(0, ref, False)
    alone.close()
    np.testing.assert_array_equal(got, ref)
