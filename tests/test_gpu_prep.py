"""The step preparation of FP64 mode (departure interpolation, extrapolated
start, ring) against the FP32-bulk mode's, which takes another path node by
node: short solves with time steps so long that the departure stencil moves by
more than a cell, on grids with one partial tile, whole tiles and a remainder,
for both interpolation orders and every payoff.

FP32-bulk solves agree with FP64 to 1e-5 relative in max-norm (the mode's bound).
"""
import numpy as np
import pytest

from conftest import gpu_solver
from paper_2511_02700_gb300.workloads import Workload, with_

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("n,steps", [(8, 6), (32, 2), (64, 6), (256, 4), (512, 3)])
@pytest.mark.parametrize("sl", [1, 3])
@pytest.mark.parametrize("payoff", [0, 1, 2])
def test_long_steps_agree_between_the_precisions(n, steps, sl, payoff):
    w = Workload("p", n=n, steps=steps, alpha=0.3, beta=(0.25, -0.3), r=0.08, tol=1e-9, sl_order=sl)
    V = {}
    for prec in ("fp64", "fp32"):
        s = gpu_solver(with_(w, precision=prec), payoff=payoff)
        _, v, _, st = s.solve(values=True)
        s.close()
        assert st == 0
        V[prec] = v.cpu().numpy()
    assert np.abs(V["fp64"] - V["fp32"]).max() <= 1e-5 * np.abs(V["fp64"]).max()
