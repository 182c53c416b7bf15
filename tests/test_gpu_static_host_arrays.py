"""pide2d_jump_static takes a field and a result by a copy where they are not memory of the
current device: pinned host arrays give the bits of device arrays, also in a captured graph, and
the entries outside the interior stay untouched."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2511_02700_gb300 import binding as B  # noqa: E402


@pytest.mark.parametrize("n", [8, 64, 256])
@pytest.mark.parametrize("host_in,host_out", [(True, False), (False, True), (True, True)])
def test_pinned_host_arrays(n, host_in, host_out):
    om = torch.rand((n, n), dtype=torch.float64, device="cuda")
    U = torch.rand((n + 1, n + 1), dtype=torch.float64, device="cuda")
    want = torch.full_like(U, -7.0)
    B.pide2d_jump_static(n, om.data_ptr(), U.data_ptr(), want.data_ptr())
    torch.cuda.synchronize()
    u = U.cpu().pin_memory() if host_in else U
    out = torch.full((n + 1, n + 1), -7.0, dtype=torch.float64)
    out = out.pin_memory() if host_out else out.cuda()
    B.pide2d_jump_static(n, om.data_ptr(), u.data_ptr(), out.data_ptr())
    torch.cuda.synchronize()
    assert torch.equal(out.cpu(), want.cpu())


def test_capture_with_device_and_pinned_arrays():
    n = 64
    om = torch.rand((n, n), dtype=torch.float64, device="cuda")
    U = torch.rand((n + 1, n + 1), dtype=torch.float64, device="cuda")
    u = U.cpu().pin_memory()
    want = torch.zeros_like(U)
    B.pide2d_jump_static(n, om.data_ptr(), U.data_ptr(), want.data_ptr())
    torch.cuda.synchronize()
    for src in (U, u):
        out = torch.zeros_like(U)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            B.pide2d_jump_static(n, om.data_ptr(), src.data_ptr(), out.data_ptr(),
                                 torch.cuda.current_stream().cuda_stream)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, want)
