"""Device memory of a problem: the dataflow sweep's face records take the bytes
of their fluxes (four directions at most: 16 bytes per column face and plane),
so a mesh that fits by its arrays' sizes can be solved."""
import pytest

from synth import phantoms as ph

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sn", [2, 4])
@pytest.mark.parametrize("L", [0, 1])
def test_face_records(sn, L):
    import torch
    from paper_1811_12391_gb300.solver import DoctorsProblem
    nx, ny, nz, G, t = 128, 128, 64, 8, 8
    p = ph.water_cylinder(nx=nx, ny=ny, nz=nz, dx=0.3, dy=0.3, dz=0.3, diameter=35.0, G=G, sn=sn, L=L)
    DoctorsProblem(p, tile=(t, t)).close()       # loads what is loaded once
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    h = DoctorsProblem(p, tile=(t, t))
    torch.cuda.synchronize()
    used = before - torch.cuda.mem_get_info()[0]
    h.close()
    GV, M = G * nx * ny * nz, (L + 1) ** 2
    faces = 8 * G * nz * 16 * ((nx // t - 1) * ny + (ny // t - 1) * nx)
    # materials and density; fluence, cross section and previous iterate (4 arrays of [G][V]), moments and sources (5 of [G][V][M])
    arrays = 5 * nx * ny * nz + 4 * GV * 4 + 5 * GV * M * 4
    assert used <= 1.1 * (arrays + faces), (used, arrays, faces)
