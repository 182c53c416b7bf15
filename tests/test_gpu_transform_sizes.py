"""Every transform length up to 2048 (each has its own number of values per
thread and units per block): the jump sum with a far field, and one iteration
of the increment loop (row DST, column solve, row DST back with the packed R2C,
column pass, inverse row pass), against the FP64 oracle at every interior node.

Tolerances as for the larger sizes: FP64 1e-12 of the scale (the weight
quadratures agree to ~1e-11 relative, the transforms to ~1e-14); FP32 1e-5 of
max |delta| for the solve and 2e-6 of sum(w) max |.| for the jump sums
(log2(P) eps_32 per transform).
"""
import numpy as np
import pytest

from paper_2511_02700_gb300.workloads import Workload, random_field

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import oracle as O  # noqa: E402
import oracle_jobs as OJ  # noqa: E402
from conftest import gpu_solver, oracle_inputs  # noqa: E402

HT, THETA = 1.0 / 64, 0.5


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("n", [8, 16, 32, 64, 128, 256, 512, 1024])
def test_each_transform_length_matches_oracle(n, precision):
    w = Workload("t", n=n, steps=64, alpha=0.5, precision=precision)
    fp64 = precision == "fp64"
    s = gpu_solver(w)
    U = random_field(n, 7 * n + 1)
    out = s.apply_jump(torch.from_numpy(U), 0.25).cpu().numpy()[1:-1, 1:-1]
    r = torch.from_numpy(OJ.probe_residual(n, n))
    d, bd, stop = s.iteration_probe(r, HT, THETA)
    s.close()
    m, g, c = oracle_inputs(w)
    pre = O.precompute(m, g, r2_order=12)
    ext = O.extend(g, c, m.r, U[1:-1, 1:-1], 0.25)
    ref = O.jump_fft(g, pre.omega, ext)
    assert np.abs(out - ref).max() <= (1e-12 if fp64 else 2e-6) * pre.sum_w * np.abs(ext).max()
    ref_d, ref_bd, ref_stop, sum_w = OJ.iteration_reference(w, n, HT, THETA, 12)
    d = d.cpu().numpy()[1:-1, 1:-1]
    bd = bd.cpu().numpy()[1:-1, 1:-1]
    dmax = np.abs(ref_d).max()
    assert np.abs(d - ref_d).max() <= (1e-12 if fp64 else 1e-5) * dmax
    assert np.abs(bd - ref_bd).max() <= (1e-12 if fp64 else 2e-6) * sum_w * dmax
    assert abs(stop - ref_stop) <= (1e-12 if fp64 else 1e-5) * ref_stop
