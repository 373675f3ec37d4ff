"""One nodal V-cycle against a model of it (paper Sec. "Numerical algorithm": the nodal projection by
multigrid): with one iteration allowed and p = 0 on entry, conjugate gradients leave p = a M b, the
V-cycle applied to the right-hand side times a = (b.z) / (z.A z).  A converged solve would hide a
wrong weight or halo of the V-cycle behind more iterations.

The model is sparse matrices in FP64: three Chebyshev steps on [1/4, 2] of D^-1 A before and after,
full weighting (the transpose of trilinear interpolation), the coarse operator from the children's
mean volume fractions, the bottom solved exactly.

Tolerance: a step's row sums 27 terms in the V-cycle's precision, 27 roundings of its unit u; a level
takes six steps, a residual and two transfers, 9 L in all on L levels.  Rounding errors of neighbouring
nodes are unrelated, so they lie in the rough part of the spectrum, which reaches down to an eighth of
its top and is amplified at most 8 times by solving: 27 x 9 L x 8 x u of |p|.
"""
import numpy as np
import pytest
import scipy.sparse as sp
import scipy.sparse.linalg as spl

import oracle as O

OUT = (O.SLIP, O.SLIP, O.SLIP, O.SLIP, O.SLIP, O.OUTFLOW)
WALLS = (O.SLIP,) * 6                     # pure Neumann: node (0, 0, 0) is held

K1 = [1.0 / 3.0, 0.0, -1.0 / 12.0, -1.0 / 12.0]   # corners that differ in 0, 1, 2, 3 coordinates


class Level:
    def __init__(self, n, h, alpha, bc):
        self.n, self.h, self.alpha = n, h, alpha          # alpha[k, j, i]
        nx, ny, nz = n
        self.shape = (nz + 1, ny + 1, nx + 1)
        node = np.arange(np.prod(self.shape)).reshape(self.shape)
        act = np.zeros(self.shape, dtype=bool)
        corner = []
        for q in range(8):
            i, j, k = q & 1, (q >> 1) & 1, q >> 2
            corner.append(node[k:k + nz, j:j + ny, i:i + nx].ravel())
            act[k:k + nz, j:j + ny, i:i + nx] |= alpha > 0
        for d in range(3):
            for hs in range(2):
                if bc[2 * d + hs] == O.OUTFLOW:
                    act[(slice(None),) * (2 - d) + (-hs,)] = False
        if O.OUTFLOW not in bc:
            act[0, 0, 0] = False
        self.act = act.ravel()
        rows, cols, vals = [], [], []
        for a in range(8):
            for b in range(8):
                w = K1[bin(a ^ b).count("1")]
                if w:
                    rows.append(corner[a])
                    cols.append(corner[b])
                    vals.append(h * w * alpha.ravel())
        A = sp.coo_matrix((np.concatenate(vals), (np.concatenate(rows), np.concatenate(cols))), shape=(node.size,) * 2)
        R = sp.diags(self.act.astype(float))
        self.A = (R @ A.tocsr() @ R + sp.diags((~self.act).astype(float))).tocsr()
        self.D = self.A.diagonal()


def hierarchy(n, h, alpha, bc):
    levels = [Level(n, h, alpha, bc)]
    while levels[-1].act.size > 125 and not any(v & 1 for v in levels[-1].n):
        f = levels[-1]
        nx, ny, nz = (v // 2 for v in f.n)
        mean = f.alpha.reshape(nz, 2, ny, 2, nx, 2).mean(axis=(1, 3, 5))
        c = Level((nx, ny, nz), 2.0 * f.h, mean, bc)
        one = []                                          # interpolation along each axis
        for v in (nz, ny, nx):
            P = sp.lil_matrix((2 * v + 1, v + 1))
            for q in range(v + 1):
                P[2 * q, q] = 1.0
                for s in (-1, 1):
                    if 0 <= 2 * q + s <= 2 * v:
                        P[2 * q + s, q] = 0.5
            one.append(P.tocsr())
        P = sp.kron(sp.kron(one[0], one[1]), one[2]).tocsr()
        f.P = sp.diags(f.act.astype(float)) @ P @ sp.diags(c.act.astype(float))
        levels.append(c)
    levels[-1].solve = spl.factorized(levels[-1].A.tocsc())
    return levels


def chebyshev(L, b, x):
    theta, delta = 0.5 * (2.0 + 0.25), 0.5 * (2.0 - 0.25)
    sigma, d = theta / delta, np.zeros_like(b)
    rho, cd, cr = 1.0 / sigma, 0.0, 1.0 / theta
    for _ in range(3):
        d = cd * d + cr * np.where(L.act, (b - L.A @ x) / L.D, 0.0)
        x = x + d
        new = 1.0 / (2.0 * sigma - rho)
        cd, cr, rho = new * rho, 2.0 * new / delta, new
    return x


def vcycle(levels, b, l=0):
    L = levels[l]
    if l + 1 == len(levels):
        return L.solve(b)
    x = chebyshev(L, b, np.zeros_like(b))
    r = np.where(L.act, b - L.A @ x, 0.0)
    return chebyshev(L, b, x + L.P @ vcycle(levels, L.P.T @ r, l + 1))


def problem(n, bc):
    h = 1.0 / n[0]
    c, r = tuple((0.5 * v + o) * h for v, o in zip(n, (0.013, 0.131, 0.272))), 0.3 * min(n) * h
    g = O.Grid(n=n, h=h, bc=bc, u_in=(0.0, 0.0, 0.0))
    geo = O.build_geometry(g, O.Shape(kind=O.SHAPE_SPHERE, p=c + (r,)))
    u = np.random.Generator(np.random.PCG64(sum(n))).uniform(-1.0, 1.0, size=(3, g.ncell))
    return g, geo, c, r, (u * (geo.alpha > 0)).ravel()


@pytest.mark.parametrize("bc", [OUT, WALLS])
@pytest.mark.parametrize("n", [(8, 8, 8), (12, 20, 28)])
def test_model(n, bc):
    """The model's operator is the oracle's, and its V-cycle contracts the error: at least threefold with an
    outflow side, as degree-3 Chebyshev smoothing on [1/4, 2] should; a held node is a point condition,
    which no coarse level represents, so there one mode goes slower (and conjugate gradients take it)."""
    g, geo, _, _, u = problem(n, bc)
    levels = hierarchy(n, g.h, geo.alpha.reshape(g.cshape()), bc)
    rng = np.random.Generator(np.random.PCG64(1))
    x = np.where(levels[0].act, rng.standard_normal(g.nnode), 0.0)
    y = O.nodal_apply(g, geo, 1.0, x)
    act = levels[0].act
    assert np.abs((levels[0].A @ x - y)[act]).max() <= 1e-13 * np.abs(y).max()
    for _ in range(30):
        e = x - vcycle(levels, np.where(act, levels[0].A @ x, 0.0))
        rate = np.sqrt((e @ (levels[0].A @ e)) / (x @ (levels[0].A @ x)))
        x = e / np.abs(e).max()
    assert rate <= (1.0 / 3.0 if bc is OUT else 1.0)


SHAPES = [(8, 8, 8),        # FP64: the finest level and the bottom in the cluster; uneven slabs
          (16, 16, 16),     # FP32: two smoothed levels in the cluster, FP64: one below the march
          (32, 32, 32),     # a level above the cluster in either precision
          (4, 8, 12), (12, 8, 4),     # five node planes: five blocks have work
          (4, 4, 32), (32, 4, 4),     # two smoothed levels of few nodes, three planes
          (12, 20, 28), (28, 20, 12), # odd bottoms, 7 planes over the blocks
          (24, 24, 8),      # three smoothed levels in the cluster (FP32)
          (40, 24, 56)]


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("bc", [OUT, WALLS])
@pytest.mark.parametrize("n", SHAPES)
def test_one_vcycle(n, bc, precision):
    import torch
    from paper_1905_07392_gb300 import ebvisc as E
    g, geo, c, r, u = problem(n, bc)
    dt = 0.01
    s = E.Solver(n, g.h, bc=bc, u_in=g.u_in, tol=1e-13, max_iters=1, precision=precision)
    s.build_sphere(c, r)
    alpha = s.geometry()["alpha"].cpu().numpy().reshape(g.cshape())
    p = torch.zeros(g.nnode, dtype=torch.float64, device="cuda:0")
    with pytest.raises(E.EbvError) as ei:
        s.solve_projection(torch.tensor(u, device="cuda:0"), p, dt)
    assert ei.value.status == next(k for k, v in E.STATUS.items() if v == "EBV_ERR_NOT_CONVERGED")
    s.close()
    levels = hierarchy(n, g.h, alpha, bc)
    b = O.nodal_rhs(g, geo, u) / dt
    z = vcycle(levels, b)
    want = (b @ z) / (z @ (levels[0].A @ z)) * z
    got = p.cpu().numpy()
    assert (got[~levels[0].act] == 0.0).all()
    tol = 27 * 9 * len(levels) * 8 * (2.0 ** -24 if precision else 2.0 ** -53)
    assert np.linalg.norm(got - want) <= tol * np.linalg.norm(want)
