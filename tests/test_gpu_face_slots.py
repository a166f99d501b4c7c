"""Face records between tiles: S2 and S4 keep theirs interleaved by plane (one
plane, odd and even numbers of planes), and a mesh of several ragged default
tiles with more planes than the fetch runs ahead, against the FP64 oracle."""
import numpy as np
import pytest

from oracle import solver as osv
from synth import phantoms as ph
from tests.parity import REL_TOL, max_rel

pytestmark = pytest.mark.gpu


def check(p, differencing, **options):
    from paper_1811_12391_gb300.solver import DoctorsProblem
    p.differencing = differencing
    sol = osv.solve(p, tol=1e-11)
    d = DoctorsProblem(p, tol=1e-6, max_iters=400, **options)
    for _ in range(2):           # the second solve uses the records handed back by the first
        d.solve()
        phi = d.fluence_host(2)
        if differencing:         # changes sign: against each group's maximum
            err = float((np.abs(phi - sol.phi) / np.abs(sol.phi).max(axis=1, keepdims=True)).max())
        else:
            err = max_rel(phi, sol.phi)
        assert err <= REL_TOL, err
    d.close()


@pytest.mark.parametrize("nz", [1, 2, 3, 4, 9, 14])
@pytest.mark.parametrize("sn,L", [(2, 0), (2, 3), (4, 1), (4, 2)])
@pytest.mark.parametrize("differencing", [0, 1])
def test_planes(nz, sn, L, differencing):
    check(ph.abdomen(nx=11, ny=9, nz=nz, d=3.0, dz=2.0, G=2, sn=sn, L=L), differencing, tile=(4, 3))


@pytest.mark.parametrize("sn,L", [(4, 0), (8, 1), (6, 2), (8, 3), (12, 3), (16, 1)])
def test_default_tiles(sn, L):
    check(ph.abdomen(nx=35, ny=19, nz=13, d=1.0, dz=1.0, G=3, sn=sn, L=L), 0)
