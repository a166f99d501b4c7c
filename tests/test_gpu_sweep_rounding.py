"""The dataflow sweep's sums keep their order: FP64 results of a solve (a mean
dose, the view weights' gradients) show the rounding of the FP32 transforms
in their last digits, so a re-ordered sum changes them.

A solve that leaves every cell one octant's contribution is reproducible to
the bit.  Photons of group 0 scatter in corner voxel A into group 1 (nowhere
else, and group 0 not at all), those of group 1 in the central voxel B into
group 2; the rest of the mesh absorbs.  Group 1 reaches the cells off A's
planes in one octant (both moment transforms, into and out of the moments
that scatter in B), group 2 the cells off B's planes in one octant each.  The gradients of the group 2 dose in the
corner opposite to A go the same way back.
"""
import os
from types import SimpleNamespace

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "sweep_rounding.npz")
N = (5, 5, 6)
B = (2, 2, 2)
CASES = [(sn, L, scheme, corner) for sn in (2, 4, 6, 8, 12, 16) for L in range(4) for scheme in (0, 1) for corner in (0, 7)]


def key(sn, L, scheme, corner):
    return f"s{sn}p{L}_{'diamond' if scheme else 'step'}_{corner}"


def problem(sn, L, scheme, corner):
    nx, ny, nz = N
    d = (1.1, 0.9, 1.3)
    lo = -0.5 * np.array([nx * d[0], ny * d[1], nz * d[2]])
    a = [0 if not corner >> ax & 1 else N[ax] - 1 for ax in range(3)]
    mat = np.zeros(N[::-1], np.uint8)
    mat[a[2], a[1], a[0]] = 1
    mat[B[2], B[1], B[0]] = 2
    st = np.array([[0.3, 0.21, 0.17], [0.9, 0.5, 0.3], [0.6, 1.1, 0.4]])
    ss = np.zeros((3, L + 1, 3, 3))
    for l in range(L + 1):
        ss[1, l, 0, 1] = 0.8 * 0.7 ** l
        ss[2, l, 1, 2] = 0.9 * 0.6 ** l
    side = np.array([1.0 if corner >> ax & 1 else -1.0 for ax in range(3)])
    pos = side * (np.abs(lo) + np.array([2.3, 3.1, 1.7]))
    src = SimpleNamespace(kind=0, pos=pos, axis=-pos / np.linalg.norm(pos), weight=3.0, spectrum=np.array([1.0, 0.0, 0.0]))
    rho = (1.0 + 0.03 * np.sin(np.arange(mat.size))).astype(np.float32)
    return SimpleNamespace(nx=nx, ny=ny, nz=nz, dx=d[0], dy=d[1], dz=d[2], origin=lo, mat=mat.reshape(-1), density=rho,
                           sigma_t=st, sigma_s=ss, sn=sn, legendre=L, sources=[src], differencing=scheme), a


def results(sn, L, scheme, corner, tile=(0, 0)):
    """Collided fluence of group 1 off A's planes and of group 2 off B's; the group 2 dose in the corner opposite to A,
    its view weight and spectrum gradients, and its density gradients off the planes of A, B and that corner."""
    import torch
    from paper_1811_12391_gb300.solver import DoctorsProblem
    p, a = problem(sn, L, scheme, corner)
    c = [n - 1 - v for n, v in zip(N, a)]
    h = DoctorsProblem(p, tol=1e-6, max_iters=50, tile=tile)
    h.solve()
    phi = h.fluence_host(1).reshape(3, *N[::-1])
    k, j, i = np.meshgrid(*(np.arange(n) for n in N[::-1]), indexing="ij")
    off = [(i != v[0]) & (j != v[1]) & (k != v[2]) for v in (a, B, c)]
    roi = np.zeros(N[::-1])
    roi[c[2], c[1], c[0]] = 1.0
    g = h.roi_gradients(np.array([[0.0, 0.0, 1.0]] * 3), torch.as_tensor(roi.reshape(-1), device="cuda"))
    density = g["density"].cpu().numpy().reshape(N[::-1])[off[0] & off[1] & off[2]]
    h.close()
    return (np.concatenate([phi[1][off[0]], phi[2][off[1]]]),
            np.concatenate([[g["J"]], g["weights"].cpu().numpy(), g["spectrum"].cpu().numpy()[:1], density[density != 0.0]]))


def check(cases):
    golden = np.load(GOLDEN)
    for c in cases:
        want = golden[key(*c)], golden[key(*c) + "_gradients"]
        assert np.count_nonzero(want[0]) > 0.9 * want[0].size
        for tile in ((0, 0), (3, 2), (10, 8), (16, 10)):
            for w, got in zip(want, results(*c, tile=tile)):
                np.testing.assert_array_equal(got.view(f"u{got.itemsize}"), w.view(f"u{w.itemsize}"),
                                              err_msg=str((key(*c), tile)))


@pytest.mark.parametrize("sn", [2, 4, 6, 8, 12, 16])
@pytest.mark.parametrize("L", [0, 1, 2, 3])
def test_bits(sn, L):
    check([c for c in CASES if c[:2] == (sn, L) and (c[2] == 0 or L in (1, 3))])


@pytest.mark.parametrize("sn", [2, 4, 6, 8, 12, 16])
@pytest.mark.parametrize("L", [0, 2])
def test_bits_diamond_denominator(sn, L):
    """P0 and P2 diamond cells: density times cross section is not rounded before the direction's term is added."""
    check([c for c in CASES if c[:2] == (sn, L) and c[2] == 1])
