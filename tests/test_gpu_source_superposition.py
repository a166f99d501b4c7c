"""The uncollided fluence of several sources is the FP32 sum, in order, of the
fluences each gives alone, to the bit, for every scattering order, with the
sources traced in chunks of all, of a few and of one, and source by source
(more materials than groups times moments)."""
import dataclasses

import numpy as np
import pytest

from synth import phantoms as ph

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("G,L,n", [(2, 0, 4), (7, 0, 6), (11, 0, 3), (4, 1, 5), (2, 2, 6), (3, 3, 4)])
def test_sum_of_single_sources(G, L, n):
    from paper_1811_12391_gb300.solver import DoctorsProblem
    p = ph.abdomen(nx=13, ny=10, nz=6, d=2.6, dz=2.0, G=G, sn=2, L=L, n_views=n)
    srcs = list(p.sources)
    srcs.insert(1, ph.Source(kind=ph.SRC_POINT, pos=np.array([3.0, -60.0, 2.0]), axis=np.array([0.0, 1.0, 0.0]), weight=0.7,
                             spectrum=srcs[0].spectrum))

    def uncollided(sources):
        h = DoctorsProblem(dataclasses.replace(p, sources=sources), tol=1e-3, max_iters=50)
        h.solve()
        phi = h.fluence_host(0)
        h.close()
        return phi

    want = np.zeros((G, p.V), np.float32)
    for s in srcs:
        want = want + uncollided([s])
    np.testing.assert_array_equal(uncollided(srcs).view(np.uint32), want.view(np.uint32))
