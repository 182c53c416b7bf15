"""The FP64 transforms run in block fixed point (one exponent per transform):
scaling of the field by powers of two from near the smallest normal to near the
largest double scales the jump sum with it, zero stays zero, and a non-finite
value reaches every output, as in floating point.

A power-of-two scale changes only exponents, so the scaled result equals the
scaled unscaled one exactly where every intermediate stays in the normal range.
"""
import numpy as np
import pytest

from conftest import gpu_solver
from paper_2511_02700_gb300.workloads import Workload, random_field

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("n", [32, 64, 256, 1024])
def test_range_and_non_finite_values(n):
    s = gpu_solver(Workload("f", n=n, steps=4, alpha=0.5, precision="fp64"))
    U = torch.from_numpy(random_field(n, n + 3, -50.0, 100.0))

    def jump(x):
        return s.apply_jump(x, 0.0, far_field=False).cpu().numpy()[1:-1, 1:-1]

    base = jump(U)
    for e in (-900, -600, 500, 900):
        assert np.array_equal(jump(U * 2.0 ** e), base * 2.0 ** e), e
    assert np.array_equal(jump(torch.zeros_like(U)), np.zeros_like(base))
    for bad in (float("nan"), float("inf")):
        V = U.clone()
        V[n // 2, n // 3] = bad
        assert not np.isfinite(jump(V)).any()
    s.close()
