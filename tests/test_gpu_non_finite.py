"""A fluence that is not finite (an emission beyond FP32) is an error on every
path that iterates, and leaves the problem fit for the next solve: on one tile,
where the sum of a group's change is NaN, and on several, where a NaN flux also
runs out the wait for a face record."""
import dataclasses

import numpy as np
import pytest

from synth import phantoms as ph
from tests.parity import REL_TOL, max_rel

pytestmark = pytest.mark.gpu

# one tile of the mesh, or several
TILES = [pytest.param((16, 16), id="one_tile"), pytest.param((4, 4), id="tiles")]


def problem(L):
    return ph.abdomen(nx=10, ny=9, nz=5, d=3.3, dz=2.0, G=3, sn=4, L=L, n_views=2)


def bad_sources(p):
    return [dataclasses.replace(s, weight=1e300) for s in p.sources]


@pytest.mark.parametrize("kernel,device_loop", [(0, 0), (0, 1), (1, 0), (3, 0), (3, 1), (5, 0)])
@pytest.mark.parametrize("L", [0, 1, 2, 3])
@pytest.mark.parametrize("tile", TILES)
def test_solve(tile, L, kernel, device_loop):
    from paper_1811_12391_gb300 import _lib as C
    from paper_1811_12391_gb300.solver import DoctorsProblem
    p = problem(L)
    h = DoctorsProblem(p, tol=1e-6, max_iters=60, tile=tile, sweep_kernel=kernel, device_loop=device_loop)
    h.solve()
    want = h.fluence_host()
    h.set_sources(bad_sources(p))
    with pytest.raises(C.DoctorsError) as e:
        h.solve()
    assert e.value.code == C.DOCTORS_ERR_INVALID_ARG
    with pytest.raises(C.DoctorsError) as e:
        h.fluence_host()
    assert e.value.code == C.DOCTORS_ERR_STATE
    h.set_sources(p.sources)
    h.solve()
    assert max_rel(h.fluence_host(), want) <= REL_TOL
    h.close()


@pytest.mark.parametrize("tile", TILES)
def test_batch_and_adjoint(tile):
    import torch
    from paper_1811_12391_gb300 import _lib as C
    from paper_1811_12391_gb300.solver import DoctorsProblem, solve_batch
    p = problem(1)
    hs = [DoctorsProblem(p, tol=1e-6, max_iters=60, tile=tile) for _ in range(3)]
    solve_batch(hs)
    want = [h.fluence_host() for h in hs]
    hs[1].set_sources(bad_sources(p))
    with pytest.raises(C.DoctorsError) as e:
        solve_batch(hs)
    assert e.value.code == C.DOCTORS_ERR_INVALID_ARG
    hs[1].set_sources(p.sources)
    solve_batch(hs)
    for h, w in zip(hs, want):
        assert max_rel(h.fluence_host(), w) <= REL_TOL
    # an adjoint response beyond FP32
    roi = torch.zeros(p.V, dtype=torch.float64, device="cuda")
    roi[p.V // 2] = 1.0
    g = hs[0].roi_gradients(p.k_dep, roi)
    with pytest.raises(C.DoctorsError) as e:
        hs[0].roi_gradients(p.k_dep, roi * 1e45)
    assert e.value.code == C.DOCTORS_ERR_INVALID_ARG
    with pytest.raises(C.DoctorsError) as e:     # the adjoint fluence of the call before is overwritten
        hs[0].fluence_host(C.DOCTORS_FLUENCE_ADJOINT)
    assert e.value.code == C.DOCTORS_ERR_STATE
    again = hs[0].roi_gradients(p.k_dep, roi)
    np.testing.assert_allclose(again["weights"].cpu().numpy(), g["weights"].cpu().numpy(), rtol=REL_TOL)
    for h in hs:
        h.close()
