"""The FP64 stopping quantity (eq. 3.25) at the ends of the number range: an increment that
overflows is not finite, and values whose squares overflow are compared as any other."""
import numpy as np
import pytest

from conftest import gpu_solver
from paper_2511_02700_gb300 import binding as B
from paper_2511_02700_gb300.workloads import Workload

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("n", [16, 64, 256])
def test_overflowing_increment_is_not_finite(n):
    # one row whose sine coefficients S_k = +-0.85e308 and their doubles are finite, while twice
    # the row itself, as the inverse transform forms it, is not: (2/n) sum |S_k sin| = 1.27 S
    k = np.arange(1, n)
    m0 = n // 3
    sin = np.sin(np.pi * np.outer(np.arange(n + 1), k) / n)
    S = np.sign(sin[m0])
    row = (2.0 / n) * sin @ S * 0.85
    assert 2.0 * 0.85 < 1.7976 < 2.0 * np.abs(row).max() and np.abs(row).max() < 1.7976
    r = np.zeros((n + 1, n + 1))
    r[n // 2] = row * 1e308
    s = gpu_solver(Workload("stop", n=n, steps=4, alpha=0.4, precision="fp64"))
    # h_t = 1e-12: the solve is the identity to 1e-6
    _, _, stop = s.iteration_probe(torch.from_numpy(r).cuda(), 1e-12, 0.5)
    s.close()
    assert not np.isfinite(stop)


def test_iteration_counts_do_not_depend_on_the_unit_of_money():
    def solve(unit, **kw):
        model = B.model_from_subordinated_bm(0.3, 0.5, (-0.1, 0.02), (0.2, 0.25), 0.3, 0.03)
        s = B.Solver(B.make_grid(64, B.PIDE2D_FP64, s0=(unit, unit)), model,
                     B.make_contract(B.PIDE2D_PUT_AVG, unit, 1.0), 8, tol=1e-10, **kw)
        price, _, stats, status = s.solve()
        s.close()
        assert status == 0
        return price / unit, stats.fp_iters_total

    price, iters = solve(1e100)
    for unit in (1e150, 1e160, 1e200, 1e250):
        p, k = solve(unit)
        assert k == iters and abs(p - price) <= 1e-12 * price
        assert solve(unit, host_loop=True) == (p, k)
