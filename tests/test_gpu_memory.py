"""Device memory of a context, which bounds the largest grid: fields of 4,194,304 nodes, so that
every array is a multiple of the allocation granularity."""
import pytest

from workloads import config

from test_gpu_parity import pkg  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
def test_fields_per_node(pkg, precision):  # noqa: F811
    torch = pytest.importorskip("torch")
    cfg = config("c1", n_elem=16, n_r=32, n_theta=64, n_phi=128)
    small = pkg.Context(*pkg.make_structs(config("c1"), precision=precision))
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    ctx = pkg.Context(*pkg.make_structs(cfg, precision=precision))
    used = free - torch.cuda.mem_get_info()[0]
    # three states of 32 variables and the filter's copy (128), primitives (7), fluxes (24), first
    # and second derivatives (63 + 66), flux divergence (8), light-cone speed, quadrature weight
    # and constraint (3), metric (9, FP64: 10), matter terms (10)
    assert ctx.n_points == 1 << 22
    assert used / (8 * ctx.n_points) < 318 + 1
    ctx.close()
    small.close()
