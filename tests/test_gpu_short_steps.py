"""The FP64 column solve for time steps so short that the implicit operator is the identity:
the increment is the residual (rounding of the sine transforms: some units of 2^-53)."""
import pytest

from conftest import gpu_solver
from paper_2511_02700_gb300.workloads import Workload, random_field

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("ht", [1e-30, 1e-120, 1e-160, 1e-300])
@pytest.mark.parametrize("n", [8, 16, 64, 256, 1024])
def test_increment_is_the_residual(n, ht):
    s = gpu_solver(Workload("short", n=n, steps=4, alpha=0.4, precision="fp64"))
    r = torch.from_numpy(random_field(n, n)).cuda()
    d, _, stop = s.iteration_probe(r, ht, 0.5)
    r, d = r[1:-1, 1:-1], d[1:-1, 1:-1]
    top = float(r.abs().max())
    assert float((d - r).abs().max()) <= 1e-13 * top
    want = float((r.abs() / r.abs().clamp(min=1.0)).max())
    assert abs(stop - want) <= 1e-13 * top
    s.close()
