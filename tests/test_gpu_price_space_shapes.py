"""The price-space jump operator on grids that PriceGrid does not give: odd and even node
counts, more price nodes than lattice points, short transforms, lattices that end above or
below x_max.  Against T_out C T_in formed densely in FP64 from the operator's own weights.

Bounds: the row and column transforms round at log2(P) units of the largest value each (FP64
1.1e-16, FP32 6e-8), T_out amplifies an axis by the sum of its weights' magnitudes.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2511_02700_gb300 import binding as B  # noqa: E402


def interpolation(nodes, t, outside):
    """Cubic Lagrange rows on the four nodes around each target; outside the nodes zero above
    (outside = 'zero'), else linear from the two end nodes."""
    n = nodes.size
    M = np.zeros((t.size, n))
    for i, v in enumerate(t):
        if outside == "zero" and v > nodes[-1]:
            continue
        if outside == "linear" and (v < nodes[0] or v > nodes[-1]):
            j = 0 if v < nodes[0] else n - 2
            d = nodes[j + 1] - nodes[j]
            M[i, j], M[i, j + 1] = (nodes[j + 1] - v) / d, (v - nodes[j]) / d
            continue
        k = min(max(int(np.searchsorted(nodes, v, side="right")) - 1, 0), n - 2)
        s = min(max(k - 1, 0), n - 4)
        for q in range(s, s + 4):
            M[i, q] = np.prod([(v - nodes[r]) / (nodes[q] - nodes[r]) for r in range(s, s + 4) if r != q])
    return M


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("nx,nz,hz,nm,npl", [
    (4, 2, 0.30, 1, 3),          # P = 16, one node pair past an odd count
    (5, 4, 0.25, 2, 6),
    (63, 4, 0.25, 2, 8),         # more price nodes than lattice points
    (64, 4, 0.25, 2, 8),
    (33, 16, 0.08, 5, 40),       # P = 128
    (32, 70, 0.02, -20, 130),    # the y_out lattice starts above 1, P = 512
    (40, 150, 0.01, 60, 480),    # P = 1024
    (21, 300, 0.004, 10, 900),   # P = 2048
])
def test_operator_matches_dense_product(nx, nz, hz, nm, npl, precision):
    x = np.concatenate(([0.0], np.cumsum(np.linspace(0.5, 1.5, nx))))
    x *= 0.9 * np.exp(npl * hz) / x[-1]
    prec = B.PIDE2D_FP64 if precision == "fp64" else B.PIDE2D_FP32_BULK
    model = B.make_model(0.4, 0.6, 1.2, (-0.1, 0.05), (0.04, 0.006, 0.06), 0.03)
    op = B.PriceJump(x, nz, hz, nm, npl, model, precision=prec)
    om = op.weights()[0].cpu().numpy()
    t_in = interpolation(x, np.exp((np.arange(-nz - nm, nz + npl) + 0.5) * hz), "zero")
    t_out = interpolation(np.exp(np.arange(-nm, npl + 1) * hz), x, "linear")
    k, P = t_out.shape[1], 1 << int(np.ceil(np.log2(max(t_in.shape[0], 4 * nz, 16))))
    V = np.random.Generator(np.random.PCG64(nx)).uniform(0.0, 100.0, (nx + 1, nx + 1))
    A = t_in @ V @ t_in.T
    C = np.fft.irfft2(np.conj(np.fft.rfft2(om, (P, P))) * np.fft.rfft2(A, (P, P)), (P, P))[:k, :k]
    ref = t_out @ C @ t_out.T
    got = op.apply(torch.from_numpy(V)).cpu().numpy()
    amp = np.abs(t_out).sum(axis=1)
    unit = (1.1e-16 if precision == "fp64" else 6e-8) * 16 * np.log2(P)
    scale = np.abs(om).sum() * np.abs(A).max()
    assert (np.abs(got - ref) <= unit * scale * np.outer(amp, amp)).all()
    op.close()
