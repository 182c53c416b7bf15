"""Creation of a pricing on the device at the sizes where its kernels change shape: the payoff's
cell averages (blocks of one, four and eight rows), the weights (a warp per integrated cell up
to a lattice of 256, one and four rows of cells a thread beyond) and the sums over them."""
import numpy as np
import pytest

import oracle as O
from conftest import gpu_solver, oracle_inputs
from oracle.scheme import initial_values, levy_density
from paper_2511_02700_gb300.workloads import Workload

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("payoff", [0, 1, 2])
@pytest.mark.parametrize("n", [8, 256, 512, 2048])
def test_initial_values_match_oracle(n, payoff):
    w = Workload("p", n=n, steps=4, alpha=0.4)
    s = gpu_solver(w, payoff=payoff)
    V = s.values().cpu().numpy()
    ref = initial_values(O.Contract(payoff, w.strike, w.maturity), O.Grid(n))
    # closed forms and smooth 20-point integrals of values up to e^2.5 S0: rounding
    assert np.abs(V - ref).max() <= 1e-12 * np.abs(ref).max()
    s.close()


@pytest.mark.parametrize("n", [8, 256, 512, 2048])
def test_weight_samples_and_rates(n):
    w = Workload("w", n=n, steps=4, alpha=0.4)
    s = gpu_solver(w)
    om, rates = s.weights()
    om, rates = om.cpu().numpy(), np.asarray(rates)
    m, g, _ = oracle_inputs(w)
    c = (np.arange(-(n // 2), n // 2) + 0.5) * g.h
    rng = np.random.Generator(np.random.PCG64(n))
    i2, i1 = rng.integers(0, n, (2, 400))
    # cells weighted by the density at their centre: beyond the zero weights and the integrated cells
    outer = np.maximum(np.abs(c[i1]), np.abs(c[i2])) > max(2.0, np.ceil(np.sqrt(0.1) * (n // 2) - 0.5)) * g.h
    want = levy_density(m, c[i1[outer]], c[i2[outer]]) * g.h ** 2
    assert outer.any() and np.abs(om[i2[outer], i1[outer]] / want - 1.0).max() < 1e-11
    inf = np.maximum(np.abs(c)[None, :], np.abs(c)[:, None]) / g.h
    assert np.array_equal(om != 0, inf > 2)
    e = np.expm1(c)
    sums = (om.sum(), (om * e[None, :]).sum(), (om * e[:, None]).sum())
    scale = np.abs(om).sum() * max(1.0, np.abs(e).max())
    assert abs(rates[0] - sums[0]) <= 1e-13 * scale
    assert abs(m.r - rates[2] - sums[1]) <= 1e-13 * scale and abs(m.r - rates[3] - sums[2]) <= 1e-13 * scale
    s.close()
