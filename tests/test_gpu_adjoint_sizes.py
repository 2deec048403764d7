"""One FP64 adjoint step on either side of the size from which a warp takes 32
nodes alone, and on ragged last groups of nodes, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_0706_0405_gb300 import lbm
from paper_0706_0405_gb300 import workloads as W
from paper_0706_0405_gb300.workloads import Side

pytestmark = pytest.mark.gpu

MIXED = (Side("outflow"), Side("reflect"),
         Side("dirichlet", "reflect", 0.05, 0.0, (1.3, 0.4, -0.2, 1.1)),
         Side("dirichlet", "outflow", 0.08, 0.5, (0.9, 0.2, 0.1, 0.8)))


@pytest.mark.parametrize("sides", [MIXED, (Side("periodic"),) * 4])
@pytest.mark.parametrize("nx,ny", [(31, 1), (8, 4), (11, 3), (152, 64), (139, 70), (157, 66)])
def test_one_adjoint_step_matches_oracle(nx, ny, sides):
    """About a hundred roundings a node, 1e-14 of the largest value, and a
    hundredfold margin; the tau derivative to 1e-12 of the sum of its terms'
    magnitudes."""
    rng = np.random.Generator(np.random.PCG64(11))
    p = W.uniform(nx, ny, (1.0, 0.0, 0.0, 1.0), dx=0.1, alpha=0.2, sides=sides, lam_scale=2.0)
    p = p.with_(tau=p.dt / 0.8)
    base = oracle.feq(p, 1.0, 0.3, -0.2, 1.0)
    f0 = base[:, None, None] * (1 + 0.1 * rng.standard_normal((9, ny, nx)))
    w = 1.0 + 0.1 * rng.standard_normal((9, ny, nx))
    with lbm.Lattice(p, "fp64") as lat:
        lat.set_f(f0, 3)
        lbm.lbm_record(lat.ctx, 1)
        lat.step(1)
        abar = w.copy()
        dtau = lbm.lbm_adjoint_step(lat.ctx, 1, abar)
    state = oracle.empty_state(p)
    oracle.interior(state)[:] = f0
    want, want_tau = oracle.adjoint_step(p, state, 3, np.pad(w, ((0, 0), (1, 1), (1, 1))))
    wi = oracle.interior(want)
    assert np.max(np.abs(abar - wi)) <= 1e-12 * np.max(np.abs(wi))
    scale = p.dt / p.tau ** 2 * np.sum(np.abs(w) * np.abs(f0))
    assert abs(dtau - want_tau) <= 1e-12 * scale
