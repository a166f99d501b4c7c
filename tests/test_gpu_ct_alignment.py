"""CT conversion on device slices: the vector form takes aligned whole fours,
the scalar one the rest and unaligned arrays; both give the oracle's bits."""
import ctypes

import numpy as np
import pytest

from oracle import ct as oct_
from synth import phantoms as ph

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 3, 4, 5, 1023, 4096 + 7])
@pytest.mark.parametrize("shift", [(0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1), (3, 2, 2)])
def test_offsets_and_tails(n, shift):
    import torch
    from paper_1811_12391_gb300 import _lib as C
    cal = ph.ct_calibration()
    rng = np.random.default_rng(n)
    hu = rng.uniform(-1500.0, 1500.0, size=n).astype(np.float32)
    hu[rng.integers(0, n, size=min(n, 8))] = np.concatenate([cal["thresholds"], cal["hu_knots"]])[:min(n, 8)]
    hu[0] = np.nan
    args = [np.ascontiguousarray(a) for a in (cal["thresholds"], cal["bin_material"], cal["hu_knots"], cal["rho_knots"])]
    m_ref, r_ref = oct_.ct_to_materials(hu, *args)
    src = torch.zeros(n + 8, device="cuda")
    src[shift[0]:shift[0] + n] = torch.as_tensor(hu, device="cuda")
    mat = torch.full((n + 8,), 99, dtype=torch.uint8, device="cuda")
    rho = torch.full((n + 8,), -1.0, device="cuda")
    f, u8 = ctypes.POINTER(ctypes.c_float), ctypes.POINTER(ctypes.c_uint8)
    C.check(C.doctors_ct_to_materials(
        ctypes.c_void_p(src.data_ptr() + 4 * shift[0]), n, args[0].size, args[0].ctypes.data_as(f),
        args[1].ctypes.data_as(u8), args[2].size, args[2].ctypes.data_as(f), args[3].ctypes.data_as(f),
        ctypes.c_void_p(mat.data_ptr() + shift[1]), ctypes.c_void_p(rho.data_ptr() + 4 * shift[2]),
        C.DOCTORS_MEM_DEVICE, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)))
    torch.cuda.synchronize()
    mat, rho = mat.cpu().numpy(), rho.cpu().numpy()
    np.testing.assert_array_equal(mat[shift[1]:shift[1] + n], m_ref)
    np.testing.assert_array_equal(rho[shift[2]:shift[2] + n].view(np.uint32), r_ref.view(np.uint32))
    assert (mat[:shift[1]] == 99).all() and (mat[shift[1] + n:] == 99).all()
    assert (rho[:shift[2]] == -1).all() and (rho[shift[2] + n:] == -1).all()
