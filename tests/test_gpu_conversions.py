"""FP32-bulk entry points round a caller's doubles to FP32 (to nearest, ties to even) and give
FP32 results back as doubles, exactly as the conversion instructions do."""
import numpy as np
import pytest

from conftest import gpu_solver
from paper_2511_02700_gb300.workloads import Workload

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("scale", [1.0, 2.0 ** -100, 2.0 ** -126, 2.0 ** -140, 2.0 ** 60])
def test_residual_is_rounded_to_nearest_even(scale):
    n = 32
    s = gpu_solver(Workload("c", n=n, steps=4, alpha=0.4, precision="fp32"))
    g = np.random.Generator(np.random.PCG64(5))
    r = g.uniform(-1.0, 1.0, (n + 1, n + 1))
    m = np.float32(r).astype(np.float64)
    half = np.abs(np.spacing(np.float32(r))).astype(np.float64) / 2
    pick = g.integers(0, 6, r.shape)
    r = np.where(pick == 0, m + half, np.where(pick == 1, m - half, np.where(pick == 2, 0.0, np.where(pick == 3, -0.0, r))))
    r = r * scale
    rounded = r.astype(np.float32).astype(np.float64)
    assert (r != rounded).any()
    got = [s.iteration_probe(torch.from_numpy(v), 0.01, 0.5) for v in (r, rounded)]
    for a, b in zip(got[0][:2], got[1][:2]):
        assert torch.equal(a, b)
        assert torch.equal(a, a.float().double())          # FP32 values, given back unchanged
    assert got[0][2] == got[1][2]
    s.close()
