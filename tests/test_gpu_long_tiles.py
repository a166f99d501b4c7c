"""Diamond sweeps of S12 P3 in tiles of one column by 224 and more, whose two
steps of face records leave no room for two steps of source records, against
the FP64 oracle."""
import numpy as np
import pytest

from oracle import solver as osv
from synth import phantoms as ph
from tests.parity import REL_TOL

pytestmark = pytest.mark.gpu


def test_long_tiles():
    from paper_1811_12391_gb300.solver import DoctorsProblem
    p = ph.abdomen(nx=11, ny=9, nz=4, d=3.0, dz=2.0, G=3, sn=12, L=3)
    p.differencing = 1
    sol = osv.solve(p, tol=1e-11)
    for tile in ((1, 224), (1, 230), (225, 1), (233, 1)):
        d = DoctorsProblem(p, tol=1e-6, max_iters=400, tile=tile)
        d.solve()
        phi = d.fluence_host(2)
        d.close()
        err = float((np.abs(phi - sol.phi) / np.abs(sol.phi).max(axis=1, keepdims=True)).max())
        assert err <= REL_TOL, (tile, err)
