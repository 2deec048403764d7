"""Step kernels at the grid sizes where their launch shape changes or their
last CTA is ragged."""
import numpy as np
import pytest

import oracle
from paper_0706_0405_gb300 import lbm
from paper_0706_0405_gb300 import workloads as W
from paper_0706_0405_gb300.workloads import Side

pytestmark = pytest.mark.gpu

PERIODIC = (Side("periodic"),) * 4
WALLS = (Side("outflow"), Side("reflect"), Side("reflect"), Side("outflow"))
INFLOW = (Side("dirichlet", state_lo=(1.0, 0.1, 0.0, 1.0)), Side("outflow"), Side("periodic"), Side("periodic"))


def _problem(nx, ny, sides, omega=0.7, steps=20):
    p = W.uniform(nx, ny, (1.0, 0.0, 0.0, 1.0), dx=0.01, alpha=0.1, sides=sides, steps=steps)
    rng = np.random.Generator(np.random.PCG64(nx * 1000 + ny))
    fields = (1.0 + 0.3 * rng.random((ny, nx)), 0.5 * rng.standard_normal((ny, nx)),
              0.5 * rng.standard_normal((ny, nx)), 1.0 + 0.3 * rng.random((ny, nx)))
    return p.with_(tau=p.dt / omega), fields


@pytest.mark.parametrize("sides", [PERIODIC, WALLS, INFLOW])
@pytest.mark.parametrize("nx,ny", [(1, 1), (31, 1), (32, 1), (33, 1), (1, 33), (5, 13), (67, 32)])
def test_fp64_step_at_the_edges_of_its_one_warp_ctas(nx, ny, sides):
    """Grids of one node, one row, one column and node counts around multiples
    of 32, after 20 steps, against the FP64 oracle at the FP64 bar: 1e-10 of
    each field's largest value (20 steps of a few hundred roundings each, at
    1.1e-16, leave three orders of magnitude)."""
    p, fields = _problem(nx, ny, sides)
    f = oracle.init(p, *fields)
    assert oracle.run(p, f, p.steps) == 0
    with lbm.Lattice(p, "fp64") as lat:
        got = [t.cpu().numpy() for t in lat.init(*fields).step(p.steps).moments()]
        assert lat.health() == 0
    for g, r in zip(got, oracle.fields(p, f)):
        assert np.max(np.abs(g - r)) <= 1e-10 * max(1.0, np.max(np.abs(r)))
