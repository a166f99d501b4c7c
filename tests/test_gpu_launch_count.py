"""doctors_result.launches counts the kernels of a solve: two for the chunk of
sources and one for their scattering, per iteration a sweep and a residual, the
next iteration's scattering source (with the zeroing of the moments in a launch
of its own where they are large), and the balance.  The loop on the device
zeroes in three launches and ends every iteration with a decision."""
import pytest

from synth import phantoms as ph

pytestmark = pytest.mark.gpu


# (mesh, launches of a scattering source): 24 MB of moments is the limit of one
@pytest.mark.parametrize("n,scatter", [(12, 1), (88, 2)])
@pytest.mark.parametrize("iters", [1, 2, 4])
def test_single_solve(n, scatter, iters):
    from paper_1811_12391_gb300.solver import DoctorsProblem
    p = ph.water_cylinder(nx=n, ny=n, nz=12, dx=0.4, dy=0.4, dz=0.4, diameter=30.0, G=5, sn=2, L=3)
    assert (16 * 5 * 12 * n * n * 4 > 24 << 20) == (scatter == 2)
    h = DoctorsProblem(p, tol=1e-6, max_iters=iters)
    h.solve(allow_not_converged=True)
    assert h.result["launches"] == 3 + 2 * iters + scatter * (iters - 1) + 1
    h.close()
    h = DoctorsProblem(p, tol=1e-6, max_iters=200)
    k = h.solve()["iterations"]                 # converged: one more iteration was enqueued
    assert 4 < k < 200 and h.result["launches"] == 3 + (2 + scatter) * (k + 1) + 1
    h.close()


@pytest.mark.parametrize("kernel,extra", [(0, 6), (5, 7)])   # split sweep: three launches, which zero the moments
def test_device_loop(kernel, extra):
    from paper_1811_12391_gb300.solver import DoctorsProblem, solve_batch
    p = ph.water_cylinder(nx=12, ny=12, nz=12, dx=2.5, dy=2.5, dz=1.0, diameter=30.0, G=5, sn=2, L=1)
    hs = [DoctorsProblem(p, tol=1e-6, max_iters=200, sweep_kernel=kernel, device_loop=1) for _ in range(3)]
    k = hs[0].solve()["iterations"]
    assert hs[0].result["launches"] == 3 + k * (extra + 1) + 1
    rs = solve_batch(hs)
    most = max(r["iterations"] for r in rs)
    assert [r["launches"] for r in rs] == [3 + most * (extra + (q == 0)) + 1 for q in range(3)]
    for h in hs:
        h.close()
