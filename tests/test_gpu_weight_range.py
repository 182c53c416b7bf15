"""Weight spectra of the FP64 column pass keep one exponent per column: the jump sum scales
exactly with the weights over the range of doubles, zero weights give zero, and a non-finite
weight reaches every output."""
import numpy as np
import pytest

from paper_2511_02700_gb300.workloads import random_field

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2511_02700_gb300 import binding as B  # noqa: E402


@pytest.mark.parametrize("n", [64, 128, 256])
def test_scaled_zero_and_non_finite_weights(n):
    U = torch.from_numpy(random_field(n, n, -50.0, 100.0)).cuda()
    om = torch.from_numpy(np.random.Generator(np.random.PCG64(n)).standard_normal((n, n))).cuda()

    def jump(w, x=U):
        out = torch.zeros_like(U)
        B.pide2d_jump_static(n, w.contiguous().data_ptr(), x.data_ptr(), out.data_ptr())
        return out[1:-1, 1:-1]

    base = jump(om)
    pad = torch.zeros((2 * n + 2, 2 * n + 2), dtype=torch.float64, device="cuda")
    pad[n // 2 + 2:3 * n // 2 + 1, n // 2 + 2:3 * n // 2 + 1] = U[1:-1, 1:-1]
    k = 2 * n - 1
    c = (-1 / 16, 9 / 16, 9 / 16, -1 / 16)
    A = sum(c[q] * pad[:, q:q + k] for q in range(4))
    A = sum(c[q] * A[q:q + k] for q in range(4))
    P = (2 * n, 2 * n)
    ref = torch.fft.irfft2(torch.conj(torch.fft.rfft2(om, s=P)) * torch.fft.rfft2(A, s=P), s=P)[1:n, 1:n]
    # four transforms of log2(2 n) roundings each, on values no larger than the norms' product
    assert float((base - ref).abs().max()) <= 4 * np.log2(2 * n) * 1.1e-16 * float(om.norm() * A.norm())
    for e in (-900, -300, 300, 900):
        assert torch.equal(jump(om * 2.0 ** e), base * 2.0 ** e), e
    assert not jump(torch.zeros_like(om)).any() and not jump(om, torch.zeros_like(U)).any()
    for bad in (float("nan"), float("inf")):
        w = om.clone()
        w[n // 3, n // 2] = bad
        assert not torch.isfinite(jump(w)).any()
