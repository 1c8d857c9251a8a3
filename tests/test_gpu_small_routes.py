"""The small form of the contractions against the large one where test_gpu_small_grids.py cannot
tell: that the two runs take different kernels, and finite states on the smallest grid."""
import math

import numpy as np
import pytest

from workloads import config

from test_gpu_parity import pkg  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

SPHERE = dict(theta_min=0.0, theta_max=math.pi, theta_basis=1)


@pytest.mark.parametrize("shape,grid,opts", [
    ((1, 4, 4, 4), {}, dict(filter=0)),                  # no filter: four nodes carry the state
    ((2, 4, 4, 4), {}, dict(filter=0, integrator=1)),
    ((1, 4, 4, 4), SPHERE, dict(filter=0)),
    ((2, 12, 12, 16), {}, {}),
    ((2, 5, 33, 10), {}, dict(glm=1, filter=0)),
])
def test_routes_differ_and_agree(pkg, shape, grid, opts):  # noqa: F811
    import torch
    from oracle import solver as so
    cfg = config("c1", n_elem=shape[0], n_r=shape[1], n_theta=shape[2], n_phi=shape[3], **grid)
    one = pkg.make_structs(cfg, **opts)
    _, _, U = so.workload_state(cfg, glm=opts.get("glm", 0))
    state = torch.from_numpy(U.reshape(-1).copy()).cuda()
    n = 3000000 // (U[0].size * sum(shape[1:])) + 1      # more nodes x lengths than the small form takes
    out, launches = [], []
    for count in (1, n):
        batch = pkg.Batch([one] * count)
        for i in range(count):
            batch.set_state(i, state, True)
        batch.step([1e-7] * count, 1)
        got = np.empty(U.size)
        batch.get_state(count - 1, got, False)
        out.append(got)
        launches.append(batch.launch_count())
        batch.close()
    assert np.isfinite(out[0]).all()
    np.testing.assert_array_equal(out[0], out[1])
    # one launch for the three directions of a list instead of one each
    assert launches[0] < launches[1]
