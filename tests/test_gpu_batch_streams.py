"""Problems of one batch on streams of their own: the loop, which runs on the
first problem's stream, starts after every problem's first-collision source."""
import pytest

from synth import phantoms as ph
from tests.parity import REL_TOL, max_rel

pytestmark = pytest.mark.gpu


def test_streams():
    import torch
    from paper_1811_12391_gb300.solver import DoctorsProblem, solve_batch
    ps = [ph.abdomen(nx=40 + 8 * q, ny=40, nz=16, d=0.8, dz=0.6, G=6, sn=4, L=1, n_views=8) for q in range(3)]
    want = []
    for p in ps:
        h = DoctorsProblem(p, tol=1e-6, max_iters=400)
        h.solve()
        want.append(h.fluence_host())
        h.close()
    hs = [DoctorsProblem(p, stream=torch.cuda.Stream(), tol=1e-6, max_iters=400) for p in ps]
    for _ in range(3):
        solve_batch(hs)
        for h, w in zip(hs, want):
            assert max_rel(h.fluence_host(), w) <= REL_TOL
    for h in hs:
        h.close()
