"""The projection hierarchy is built in the precision the solves use, once: its FP64 inverse diagonals
and its bottom inverse lie where the FP32 ones do, so a hierarchy of the other precision cannot be
kept beside it.  A change of precision builds it anew, and the steps are those of a context created
with that precision, bit for bit."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _context(E, precision, n=(12, 10, 14)):
    h = 1.0 / n[0]
    s = E.Solver(n, h, tol=1e-11, max_iters=500, precision=precision, tau0=2.0, m=1e3, bi_cfl=0.5)
    s.build_spheres([[0.51 * n[0] * h, 0.53 * n[1] * h, 0.56 * n[2] * h, 0.3 * min(n) * h]])
    return s


def _step(s):
    rng = np.random.Generator(np.random.PCG64(6))
    u = rng.uniform(-1e-3, 1e-3, size=(3, s.ncell))
    u[2] += 1.0
    alpha = s.geometry()["alpha"].cpu().numpy()
    u = torch.tensor((u * (alpha > 0)).ravel(), device=DEV)
    p = torch.zeros(s.nnode, dtype=torch.float64, device=DEV)
    st = s.advance(u, p)
    return u, p, st["iters"]


@pytest.mark.parametrize("start,then", [(0, 1), (1, 0)])
def test_one_hierarchy_per_precision(start, then):
    from paper_1905_07392_gb300 import ebvisc as E
    s, fresh = _context(E, start), _context(E, then)
    _step(s)
    s.profile_begin()
    s.set_params(precision=then)
    k = s.profile_end()
    # two bottom inverses: the projection's and the nodal one's (the viscous ones follow the viscosity)
    assert k["k_gj_first"]["launches"] == 2
    (u, p, it), (uf, pf, itf) = _step(s), _step(fresh)
    assert torch.equal(u, uf) and torch.equal(p, pf) and it == itf
    s.close()
    fresh.close()
