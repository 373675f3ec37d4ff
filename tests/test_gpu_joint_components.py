"""The three viscous systems run side by side, and each component's result and iterations are those it
has alone (paper Eq. implicit-viscous): the same bits whatever the other two solve for, whether they
end earlier, later, or at once (a zero right-hand side, which is solved by zero)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
SHAPES = [(16, 16, 16),    # every level in the cluster kernel
          (24, 20, 28), (40, 24, 56),
          (64, 64, 64),    # fused sweeps or colour passes above the cluster
          (128, 96, 96)]   # enough cells that ended components are skipped in every kernel


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n", SHAPES)
def test_components_do_not_meet(n, precision):
    from paper_1905_07392_gb300 import ebvisc as E
    h = 1.0 / n[0]
    # two slip sides, two no-slip sides, inflow at rest and outflow: three different diagonals, and a
    # right-hand side that is exactly zero where psi is
    s = E.Solver(n, h, bc=(E.SLIP, E.SLIP, E.NOSLIP, E.NOSLIP, E.INFLOW, E.OUTFLOW), u_in=(0.0, 0.0, 0.0), tol=1e-10,
                 max_iters=500, precision=precision, tau0=2.0, m=1e3, bi_cfl=0.5)
    s.build_spheres([[0.5 * n[0] * h, 0.51 * n[1] * h, 0.52 * n[2] * h, 0.27 * min(n) * h]])
    alpha = s.geometry()["alpha"]
    rng = np.random.Generator(np.random.PCG64(sum(n)))
    x, y, z = np.meshgrid(*[np.arange(v) * h for v in n[::-1]], indexing="ij")[::-1]
    psi = np.stack([np.cos(3.0 * x) * (1.0 + y * z), rng.uniform(-1.0, 1.0, x.shape), np.zeros(x.shape)])
    psi[2, n[2] - 2, n[1] // 3, 1] = 1.0
    psi = torch.tensor(psi.reshape(3, -1), device=DEV) * (alpha > 0)
    eta = torch.tensor(rng.uniform(1.0, 50.0, s.ncell), device=DEV)
    dt = 0.2 * h * h

    def solve(which):
        p = torch.zeros_like(psi)
        for q in which:
            p[q] = psi[q]
        ut = torch.full((3 * s.ncell,), 7.0, dtype=torch.float64, device=DEV)
        st = s.solve_viscous(eta, p.reshape(-1).contiguous(), dt, ut)
        assert max(st["res"][1:4]) <= 1e-10
        return ut.reshape(3, -1), st["iters"][1:4]

    alone = [solve([q]) for q in range(3)]
    for q in range(3):
        assert alone[q][1][q] > 0
    for which in ([0, 1, 2], [0, 1], [1, 2], [0, 2]):
        ut, it = solve(which)
        for q in range(3):
            if q in which:
                assert torch.equal(ut[q], alone[q][0][q]) and it[q] == alone[q][1][q], (which, q)
            else:
                assert not ut[q].any() and it[q] == 0, (which, q)
    s.close()
