"""One step against the oracle on grids of many shapes (paper Algorithm 1): the
solver kernels choose their form by the grid -- one level or several, levels
within one block, odd and even row lengths, odd bottoms, sizes that are or are
not multiples of 8 and 16 -- and every choice must give the oracle's step.
The tolerance is that of the other parity tests: both sides solve to 1e-13,
and a relative residual of 1e-13 bounds u and p to 1e-10.  The captured step
(advance_graph) must give the eager step's result bit for bit.  The sphere's
centre is off the grid's centre by another amount along each axis: with equal
offsets the two largest components of the wall normal are equal in many cut
cells, and which of them Eq. dudn then takes as its axis is decided by the last
bit of the geometry.
"""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
SHAPES = [(5, 3, 7),      # a single level, odd rows
          (6, 4, 10),     # two levels, bottom 3 x 2 x 5
          (14, 14, 14),   # bottom 7^3 = 343 unknowns, 512 nodes
          (12, 10, 14),   # every level within one block
          (16, 16, 16), (32, 32, 32),
          (20, 12, 28),   # odd half-rows on level 1
          (24, 20, 28),   # nx a multiple of 8 but not of 16
          (48, 16, 32),   # a multiple of 16, flat
          (40, 24, 56),   # a multiple of 8, odd bottom
          (2, 6, 3), (2, 2, 3)]   # too few cells to hold three components' vectors: solved one after another


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n", SHAPES)
def test_step_matches_oracle(n, precision):
    from paper_1905_07392_gb300 import ebvisc as E
    h = 1.0 / n[0]
    c = tuple((0.5 * v + o) * h for v, o in zip(n, (0.013, 0.131, 0.272)))
    r = 0.3 * min(n) * h
    kw = dict(rho=1.0, mu=1.0, tau0=2.0, m=1e3, bi_cfl=0.5)
    s = E.Solver(n, h, tol=1e-13, max_iters=5000, precision=precision, **kw)
    s.build_sphere(c, r)
    g = O.Grid(n=n, h=h)
    geo = O.build_geometry(g, O.Shape(kind=O.SHAPE_SPHERE, p=c + (r,)))
    P = O.Params(tol=1e-13, max_iters=200000, **kw)
    rng = np.random.Generator(np.random.PCG64(n[0]))
    u0 = rng.uniform(-1e-3, 1e-3, size=(3, g.ncell))
    u0[2] += 1.0
    u0 = (u0 * (geo.alpha > 0)).ravel()
    uo, po, sto = O.advance(g, geo, P, u0, np.zeros(g.nnode))
    u, p = torch.tensor(u0, device=DEV), torch.zeros(g.nnode, dtype=torch.float64, device=DEV)
    st = s.advance(u, p)
    assert st["dt"] == pytest.approx(sto["dt"], rel=1e-12)
    assert np.linalg.norm(u.cpu().numpy() - uo) <= 1e-10 * np.linalg.norm(uo)
    assert np.linalg.norm(p.cpu().numpy() - po) <= 1e-10 * np.linalg.norm(po)
    ug, pg = torch.tensor(u0, device=DEV), torch.zeros(g.nnode, dtype=torch.float64, device=DEV)
    sg = s.advance_graph(ug, pg, steps=1)
    assert torch.equal(u, ug) and torch.equal(p, pg)
    assert sg["iters"] == st["iters"]
    s.close()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n", [(16, 16, 16), (32, 32, 32), (24, 20, 28), (12, 12, 24), (32, 32, 4), (64, 64, 8),
                               (48, 40, 56), (64, 64, 64)])
def test_vcycle_contracts(n, precision):
    """A fault in the coarse end of the V-cycle (slabs of one or two levels over a cluster, split
    along z or y, even or uneven, with or without a level every block smooths itself) leaves the
    solution right and only costs iterations.  Two red-black sweeps each way reduce the error of
    these operators at least threefold per CG iteration, so 1e-12 takes at most
    log(1e12) / log(3) = 25.2 iterations."""
    from paper_1905_07392_gb300 import ebvisc as E
    h = 1.0 / n[0]
    s = E.Solver(n, h, tol=1e-12, max_iters=500, precision=precision, tau0=2.0, m=1e3, bi_cfl=0.5)
    s.build_spheres([[0.5 * n[0] * h, 0.51 * n[1] * h, 0.52 * n[2] * h, 0.27 * min(n) * h]])
    rng = np.random.Generator(np.random.PCG64(n[2]))
    u0 = rng.uniform(-1e-3, 1e-3, size=(3, s.ncell))
    u0[2] += 1.0
    alpha = s.geometry()["alpha"].cpu().numpy()
    u = torch.tensor((u0 * (alpha > 0)).ravel(), device=DEV)
    st = s.advance(u, torch.zeros(s.nnode, dtype=torch.float64, device=DEV))
    it = st["iters"]
    assert max(it[:4] + it[5:9]) <= 26, it   # (slots 4 and 9 are the nodal solves)
    assert max(st["res"]) <= 1e-12
    s.close()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n", [(2, 2, 2), (4, 2, 6), (36, 20, 28), (64, 16, 32), (32, 8, 8)])
def test_nodal_projection_matches_oracle(n, precision):
    """The nodal passes march tiles of 32 x 8 interior nodes and list the rest: no interior, one
    node, partial tiles, exactly full ones.  Both sides solve to 1e-13 (see above for the bound)."""
    from paper_1905_07392_gb300 import ebvisc as E
    h = 1.0 / n[0]
    c, r = tuple((0.5 * v + 0.1) * h for v in n), 0.3 * min(n) * h
    s = E.Solver(n, h, tol=1e-13, max_iters=5000, precision=precision)
    s.build_sphere(c, r)
    g = O.Grid(n=n, h=h)
    geo = O.build_geometry(g, O.Shape(kind=O.SHAPE_SPHERE, p=c + (r,)))
    P = O.Params(tol=1e-13, max_iters=200000)
    rng = np.random.Generator(np.random.PCG64(n[0] + n[1]))
    ut0 = (rng.uniform(-0.1, 0.1, size=(3, g.ncell)) * (geo.alpha > 0)).ravel()
    p0 = rng.uniform(-1.0, 1.0, size=g.nnode)
    dt = 0.01
    uo, po = O.nodal_project(g, geo, P, dt, ut0.copy(), p0.copy())[:2]
    u, p = torch.tensor(ut0, device=DEV), torch.tensor(p0, device=DEV)
    s.solve_projection(u, p, dt)
    assert np.linalg.norm(u.cpu().numpy() - uo) <= 1e-10 * np.linalg.norm(uo)
    assert np.linalg.norm(p.cpu().numpy() - po) <= 1e-10 * np.linalg.norm(po)
    s.close()
