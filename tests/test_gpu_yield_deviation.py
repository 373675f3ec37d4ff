"""The yield-stress deviation eta ||g|| / tau0 - 1 at yield stresses whose reciprocal overflows or
is subnormal, beside an ordinary one, against the oracle's division."""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("moving", [False, True])
@pytest.mark.parametrize("tau0", [1e-320, 1e-309, 3e-308, 0.7, 1e308])
def test_yield_deviation(tau0, moving):
    from paper_1905_07392_gb300 import ebvisc as E
    n = 8
    # (a power law of index 1: the stress is mu ||g||, of the order of tau0, whatever tau0 is)
    kw = dict(tau0=tau0, m=1e2, n_flow=1.0, mu=min(tau0, 1e305))
    s = E.Solver((n, n, n), 1.0 / n, model=E.POWER_LAW, **kw)
    s.build_sphere((0.5, 0.47, 0.53), 0.2)
    g = O.Grid(n=(n, n, n), h=1.0 / n)
    geo = O.build_geometry(g, O.Shape(kind=O.SHAPE_SPHERE, p=(0.5, 0.47, 0.53, 0.2)))
    u = np.random.Generator(np.random.PCG64(5)).uniform(-1.0, 1.0, size=(3, g.ncell)) * float(moving)
    u = (u * (geo.alpha > 0)).ravel()
    _, want = O.flow_diagnostics(g, geo, O.Params(model=O.POWERLAW, **kw), u)
    lam, dev = (torch.empty(g.ncell, dtype=torch.float64, device="cuda:0") for _ in range(2))
    s.flow_diagnostics(torch.tensor(u, device="cuda:0"), lam, dev)
    s.close()
    # a subnormal stress of q units in the last place is off by at most one: 1e-320 is 2024 of them
    tol = 1e-12 + 2.0 * 5e-324 / tau0
    assert np.isfinite(want).all()
    assert (np.abs(dev.cpu().numpy() - want) <= tol * (1.0 + np.abs(want))).all()
