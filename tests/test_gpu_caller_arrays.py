"""Caller arrays are read and written in place where they are memory of the
current device aligned to their elements, and staged otherwise: host arrays and
misaligned device arrays give the same bits, and entries outside the interior
stay untouched where the entry point says so."""
import numpy as np
import pytest

from conftest import gpu_solver
from paper_2511_02700_gb300.workloads import Workload, random_field

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2511_02700_gb300 import binding as B  # noqa: E402


def misaligned(x):
    """A device copy of x that starts 4 bytes past an 8-byte boundary: (owner, pointer)."""
    buf = torch.zeros(x.numel() * 8 + 16, dtype=torch.uint8, device="cuda")
    buf[4:4 + x.numel() * 8] = x.contiguous().view(torch.uint8).reshape(-1)
    return buf, buf.data_ptr() + 4


def read_back(buf, like):
    return buf[4:4 + like.numel() * 8].clone().view(torch.float64).reshape(like.shape).cpu().numpy()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("n", [8, 64])
def test_host_device_and_misaligned_arrays_agree(n, precision):
    s = gpu_solver(Workload("a", n=n, steps=4, alpha=0.4, precision=precision))
    U = random_field(n, n)
    dev = torch.from_numpy(U).cuda()
    fill = torch.full_like(dev, -7.0)

    out_d = fill.clone()
    B.pide2d_apply_jump(s.h, dev.data_ptr(), 0.3, 1, out_d.data_ptr())
    out_h = np.full_like(U, -7.0)
    B.pide2d_apply_jump(s.h, U.ctypes.data, 0.3, 1, out_h.ctypes.data)
    ib, ip = misaligned(dev)
    ob, op = misaligned(fill)
    B.pide2d_apply_jump(s.h, ip, 0.3, 1, op)
    ref = out_d.cpu().numpy()
    assert np.array_equal(ref, out_h) and np.array_equal(ref, read_back(ob, fill))
    ring = np.ones_like(U, dtype=bool)
    ring[1:-1, 1:-1] = False
    assert (ref[ring] == -7.0).all()
    same = dev.clone()                                  # in place: input and output are one array
    B.pide2d_apply_jump(s.h, same.data_ptr(), 0.3, 1, same.data_ptr())
    assert np.array_equal(same.cpu().numpy()[1:-1, 1:-1], ref[1:-1, 1:-1])

    dd, bd = fill.clone(), fill.clone()
    st = B.pide2d_iteration_probe(s.h, dev.data_ptr(), 0.01, 0.5, dd.data_ptr(), bd.data_ptr())
    dh, bh = np.full_like(U, -7.0), np.full_like(U, -7.0)
    assert st == B.pide2d_iteration_probe(s.h, U.ctypes.data, 0.01, 0.5, dh.ctypes.data, bh.ctypes.data)
    assert np.array_equal(dd.cpu().numpy(), dh) and np.array_equal(bd.cpu().numpy(), bh)
    assert (dh[ring] == -7.0).all()

    vd, vh = torch.empty_like(dev), np.empty_like(U)
    vb, vp = misaligned(fill)
    for p in (vd.data_ptr(), vh.ctypes.data, vp):
        B.pide2d_get_values(s.h, p)
    assert np.array_equal(vd.cpu().numpy(), vh) and np.array_equal(vh, read_back(vb, fill))
    gd, gh = fill.clone(), np.full_like(U, -7.0)
    B.pide2d_greeks(s.h, gd.data_ptr(), None, None, None, None)
    B.pide2d_greeks(s.h, gh.ctypes.data, None, None, None, None)
    assert np.array_equal(gd.cpu().numpy(), gh)
    s.close()


@pytest.mark.parametrize("n", [8, 64])
def test_static_jump_with_misaligned_arrays(n):
    om = torch.rand((n, n), dtype=torch.float64, device="cuda")
    U = torch.rand((n + 1, n + 1), dtype=torch.float64, device="cuda")
    out = torch.zeros_like(U)
    B.pide2d_jump_static(n, om.data_ptr(), U.data_ptr(), out.data_ptr())
    ub, up = misaligned(U)
    ob, op = misaligned(torch.zeros_like(U))
    B.pide2d_jump_static(n, om.data_ptr(), up, op)
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy(), read_back(ob, U))
