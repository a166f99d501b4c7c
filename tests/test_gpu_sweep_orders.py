"""Parity of the dataflow sweep over angular and scattering orders: every set of
directions (pairs under the exchange of x and y, single ones) with every number
of moments, on meshes with ragged tiles, small (one face warp, two column
warps) and large, step and diamond, against the FP64 oracle."""
import numpy as np
import pytest

from oracle import solver as osv
from synth import phantoms as ph
from tests.parity import REL_TOL, max_rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sn", [2, 4, 6, 8, 12, 16])
@pytest.mark.parametrize("L", [0, 1, 2, 3])
def test_orders(sn, L):
    from paper_1811_12391_gb300.solver import DoctorsProblem
    p = ph.abdomen(nx=11, ny=9, nz=3, d=3.0, dz=2.0, G=3, sn=sn, L=L)
    for differencing in (0, 1):
        p.differencing = differencing
        sol = osv.solve(p, tol=1e-11)
        for tile in ((0, 0), (5, 3), (16, 8)):
            d = DoctorsProblem(p, tol=1e-6, max_iters=400, tile=tile)
            d.solve()
            phi = d.fluence_host(2)
            d.close()
            if differencing:     # changes sign: against each group's maximum
                err = float((np.abs(phi - sol.phi) / np.abs(sol.phi).max(axis=1, keepdims=True)).max())
            else:
                err = max_rel(phi, sol.phi)
            assert err <= REL_TOL, (sn, L, differencing, tile, err)
