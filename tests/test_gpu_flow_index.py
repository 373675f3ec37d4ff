"""Apparent viscosity at every flow index the power law treats apart (paper Table "Generalised
Newtonian fluid models": n - 1 in quarters takes square roots) and at one it does not, against
the oracle's pow.  Both sides are FP64 formulas of a few roundings each: 1e-12 as in the other
viscosity tests."""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model", ["HERSCHEL_BULKLEY", "POWER_LAW"])
@pytest.mark.parametrize("n_flow", [0.0, 0.25, 0.5, 0.75, 1.0, 1.25, 1.5, 1.75, 2.0, 1.1, 2.25])
def test_flow_index(n_flow, model):
    from paper_1905_07392_gb300 import ebvisc as E
    n = 16
    kw = dict(tau0=0.7, m=1e2, n_flow=n_flow, mu=1.3)
    s = E.Solver((n, n, n), 1.0 / n, model=getattr(E, model), **kw)
    s.build_sphere((0.5, 0.47, 0.53), 0.2)
    g = O.Grid(n=(n, n, n), h=1.0 / n)
    geo = O.build_geometry(g, O.Shape(kind=O.SHAPE_SPHERE, p=(0.5, 0.47, 0.53, 0.2)))
    rng = np.random.Generator(np.random.PCG64(3))
    u = rng.uniform(-1.0, 1.0, size=(3, g.ncell)) * 10.0 ** rng.uniform(-6.0, 0.0, size=g.ncell)
    u = (u * (geo.alpha > 0)).ravel()
    eta_o, sr_o = O.strain_eta(g, geo, O.Params(model=getattr(O, "HB" if model == "HERSCHEL_BULKLEY" else "POWERLAW"), **kw), u)
    eta = torch.empty(g.ncell, dtype=torch.float64, device="cuda:0")
    sr = torch.empty_like(eta)
    s.update_viscosity(torch.tensor(u, device="cuda:0"), eta, sr)
    assert (np.abs(sr.cpu().numpy() - sr_o) <= 1e-12 * np.abs(sr_o).max()).all()
    assert (np.abs(eta.cpu().numpy() - eta_o) <= 1e-12 * np.abs(eta_o)).all()
    s.close()
