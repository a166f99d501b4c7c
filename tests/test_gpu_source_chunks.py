"""First-collision source of several sources traced in chunks: chunk sizes of
one, a few and all sources, with collimated, isotropic and volume sources mixed,
and more materials than a chunk's buffer holds (source by source)."""
import dataclasses

import numpy as np
import pytest

from oracle import solver as osv
from synth import phantoms as ph
from tests.parity import REL_TOL, max_rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("G,L,n", [(2, 0, 3), (5, 0, 4), (3, 1, 5), (2, 2, 2), (3, 3, 1), (11, 0, 5)])
def test_chunked_sources(G, L, n):
    from paper_1811_12391_gb300.solver import DoctorsProblem
    p = ph.abdomen(nx=10, ny=9, nz=4, d=3.3, dz=2.0, G=G, sn=4, L=L, n_views=n)
    spec = p.sources[0].spectrum
    srcs = list(p.sources)
    srcs.insert(1, ph.Source(kind=ph.SRC_VOLUME, pos=np.zeros(3), axis=np.array([0.0, 0.0, 1.0]), weight=1e-5, spectrum=spec))
    srcs.append(ph.Source(kind=ph.SRC_POINT, pos=np.array([3.0, -60.0, 2.0]), axis=np.array([0.0, 1.0, 0.0]), weight=0.7,
                          spectrum=spec))
    p = dataclasses.replace(p, sources=srcs)
    sol = osv.solve(p, tol=1e-11)
    d = DoctorsProblem(p, tol=1e-6, max_iters=400)
    for _ in range(2):          # the buffers of the first solve are used again
        d.solve()
        assert max_rel(d.fluence_host(0), sol.phi_u) <= REL_TOL
        assert max_rel(d.fluence_host(2), sol.phi) <= REL_TOL
    d.close()
