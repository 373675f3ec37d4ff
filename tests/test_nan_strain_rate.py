"""A velocity that is not a number leaves the strain rate of the cells around it undefined; the
viscosity laws then take their limits at rest, as the oracle's comparisons do (paper Table
"Generalised Newtonian fluid models"), and Lambda is 0.  Both signs of NaN: an integer comparison
that orders patterns like numbers tells them apart.  Beside it a CPU model of that comparison
(gt_nonneg, ebv_internal.cuh) at the edges of every range.
"""
import numpy as np
import pytest

import oracle as O


def test_integer_comparison():
    """gt_nonneg's integer steps on every pair of edge values (b not negative and not NaN) against a > b."""
    v = np.array([0.0, 5e-324, 1e-310, np.finfo(float).tiny, 1e-2, 40.0, np.nextafter(40.0, 41.0), 1e308, np.inf, np.nan])
    a, b = (q.ravel() for q in np.meshgrid(np.concatenate([v, -v]), v[:-1]))
    ua, ub = np.ascontiguousarray(a).view(np.uint64), np.ascontiguousarray(b).view(np.uint64)
    got = ua - ub - np.uint64(1) < np.uint64(0x7ff0000000000000) - ub
    with np.errstate(invalid="ignore"):
        assert (got == (a > b)).all()


@pytest.mark.gpu
@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("model,n_flow", [("NEWTONIAN", 1.0), ("BINGHAM", 1.0), ("HERSCHEL_BULKLEY", 0.5),
                                          ("HERSCHEL_BULKLEY", 1.1), ("POWER_LAW", 0.75)])
def test_viscosity_next_to_nan(model, n_flow, sign):
    import torch
    from paper_1905_07392_gb300 import ebvisc as E
    n = 16
    kw = dict(tau0=0.7, m=1e2, n_flow=n_flow, mu=1.3)
    s = E.Solver((n, n, n), 1.0 / n, model=getattr(E, model), **kw)
    s.build_sphere((0.5, 0.47, 0.53), 0.2)
    g = O.Grid(n=(n, n, n), h=1.0 / n)
    geo = O.build_geometry(g, O.Shape(kind=O.SHAPE_SPHERE, p=(0.5, 0.47, 0.53, 0.2)))
    rng = np.random.Generator(np.random.PCG64(4))
    u = rng.uniform(-1.0, 1.0, size=(3, g.ncell)) * (geo.alpha > 0)
    at = [(8, 8, 14), (0, 5, 3), (15, 15, 15)]           # inside, at a side, at a corner
    for q, (i, j, k) in enumerate(at):
        u[q, (k * n + j) * n + i] = np.copysign(np.nan, sign)
    om = {"NEWTONIAN": O.NEWTONIAN, "BINGHAM": O.BINGHAM, "HERSCHEL_BULKLEY": O.HB, "POWER_LAW": O.POWERLAW}[model]
    eta_o, sr_o = O.strain_eta(g, geo, O.Params(model=om, **kw), u.ravel())
    ud = torch.tensor(u.ravel(), device="cuda:0")
    out = [torch.empty(g.ncell, dtype=torch.float64, device="cuda:0") for _ in range(4)]
    s.update_viscosity(ud, out[0], out[1])
    s.flow_diagnostics(ud, out[2], out[3])
    s.close()
    eta, sr, lam, dev = (t.cpu().numpy() for t in out)
    bad = np.isnan(sr_o)
    assert bad.sum() >= 6 and (np.isnan(sr) == bad).all()
    assert np.isfinite(eta_o).all()
    # (FP64 formulas of a few roundings on either side: 1e-12 as in the other viscosity tests)
    assert (np.abs(eta - eta_o) <= 1e-12 * np.abs(eta_o)).all()
    assert (lam[bad] == 0.0).all() and np.isnan(dev[bad]).all()
    assert np.isfinite(lam[~bad]).all() and np.isfinite(dev[~bad]).all()
