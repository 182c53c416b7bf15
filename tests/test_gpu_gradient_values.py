"""The adjoint's gradient for drifts at and near zero stays at the values it has always had.

The weights' derivatives are differences of two precomputes as little as 1e-8 apart, so a change
of rounding in the density, or of the order in which cells are summed, moves a drift component by
1e-9 to 1e-8.  The values are those of the Lagrange form of the density summed in storage order;
the bound is that of an FP64 result, 1e-9 of the largest component."""
import numpy as np
import pytest

from paper_2511_02700_gb300 import binding as B

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

# (n, beta): d price / d (sigma1, sigma2, corr, kappa, beta1, beta2)
KEPT = {
    (128, (0.0, 0.0)): (14.243082307827647, 15.66309827298288, 2.4332816625267455, -0.6270322260777608,
                        0.7655177182392069, 1.022948129747223),
    (128, (-0.14, 2e-4)): (12.728049041513183, 14.844236711118723, 2.340828933103938, -0.3865427806434314,
                           -2.4933472436390134, -2.2364507325550105),
    (256, (1e-3, -1e-3)): (14.27009386244343, 15.684766738768884, 2.4449725643249574, -0.6318866364071246,
                           0.7738065234160636, 1.0189349450644873),
}


@pytest.mark.parametrize("n,beta", list(KEPT))
def test_drift_gradient_keeps_its_values(n, beta):
    w = (0.3, 0.5, beta, (0.2, 0.25), 0.3, 0.03)
    s = B.Solver(B.make_grid(n, B.PIDE2D_FP64), B.model_from_subordinated_bm(*w),
                 B.make_contract(B.PIDE2D_PUT_AVG, 100.0, 1.0), n // 8, tol=1e-10)
    s.record(interval=8, ndirs=6)
    s.solve()
    g, status = s.adjoint(B.subordinated_bm_directions(*w[:5]))
    s.close()
    want = np.array(KEPT[n, beta])
    assert status == 0 and np.abs(np.array(g) - want).max() <= 1e-9 * np.abs(want).max(), g
