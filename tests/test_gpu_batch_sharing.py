"""Batches whose dataflow sweeps share the CTA slots and batches whose sweeps
do not (large direction tables, or enough tasks to fill the slots many times):
the same fluences as the instances' own solves, and no more time than these."""
import pytest

from synth import phantoms as ph
from tests.parity import REL_TOL, max_rel

pytestmark = pytest.mark.gpu


def solvers(n, nx, ny, nz, sn, L, G):
    from paper_1811_12391_gb300.solver import DoctorsProblem
    return [DoctorsProblem(ph.water_cylinder(nx=nx + 4 * q, ny=ny, nz=nz, dx=35.2 / nx, dy=35.2 / ny, dz=0.5, diameter=35.0 - q, G=G,
                                             sn=sn, L=L), tol=1e-6, max_iters=400) for q in range(n)]


@pytest.mark.parametrize("sn,L", [(4, 0), (8, 2), (8, 3), (12, 1), (16, 1)])
def test_results(sn, L):
    from paper_1811_12391_gb300.solver import solve_batch
    hs = solvers(3, 28, 20, 9, sn, L, 5)
    want = []
    for h in hs:
        h.solve()
        want.append(h.fluence_host())
    solve_batch(hs)
    for h, w in zip(hs, want):
        assert max_rel(h.fluence_host(), w) <= REL_TOL
        h.close()


def test_no_slower_than_single_solves():
    """S8 P3, 19 groups, 64x64x32: 8 % faster than one by one; sharing the slots 7 % slower."""
    from paper_1811_12391_gb300.solver import solve_batch
    hs = solvers(4, 64, 64, 32, 8, 3, 19)
    single = min(sum(h.solve()["ms_total"] for h in hs) for _ in range(3))
    batch = min(solve_batch(hs)[0]["ms_total"] for _ in range(3))
    assert batch <= single, (batch, single)
    for h in hs:
        h.close()
