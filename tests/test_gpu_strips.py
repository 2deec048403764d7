"""Batches of thin problems advanced with whole columns in registers
(temporal blocking of two- and four-row problems) against each problem
stepped alone: the same operations node by node, so the same bits."""
import numpy as np
import pytest

from paper_0706_0405_gb300 import lbm
from paper_0706_0405_gb300 import workloads as W

pytestmark = pytest.mark.gpu

P, O, R = W.Side("periodic"), W.Side("outflow"), W.Side("reflect")
D = W.Side("dirichlet", state_lo=(1.2, 0.3, 0.1, 1.1))
DX = 0.01


def _split(speed):
    """Fixed state below the split, outflow above; the split climbs over the
    rows during the run."""
    return W.Side("dirichlet", "outflow", 0.5 * DX, speed, state_lo=(1.1, 0.2, 0.0, 1.2))


# Widths around a warp's 30 stored columns, a window's edges (4 warps: 122
# columns, 114 stored at a problem's end and 108 between) and the smallest grids.
WIDTHS = [1, 2, 3, 15, 29, 30, 31, 32, 61, 107, 108, 109, 114, 115, 119, 120, 121, 122, 223, 256, 700]


def _problems(rows):
    st = (1.0, 0.3, 0.05, 1.0)
    sides = [(O, O), (R, O), (D, R), (_split(20.0), D), (R, _split(30.0))]
    return [W.uniform(nx, rows, st, dx=DX, sides=sides[k % len(sides)] + (P, P)) for k, nx in enumerate(WIDTHS)]


@pytest.mark.parametrize("rows", [2, 4])
@pytest.mark.parametrize("prec", ["fp32", "fp32_t64", "fp32_tdf", "fp32_cons"])
def test_columns_in_registers_equal_problems_stepped_alone(prec, rows):
    probs = _problems(rows)
    fields = [W.initial_fields(p, seed=k, sigma=0.01) for k, p in enumerate(probs)]
    with lbm.Batch(probs, prec) as b:
        b.init(fields).set_launch(1, 0, 7).step(30).step(2).set_launch(1, 3, 5).step(11)
        # the tile kernel reads the ghost cells the strips left
        b.set_launch(2, 0, 0).step(3).set_launch(1, 0, 3).step(14)
        b.sync()
        got = [b.get_f(k).cpu().numpy() for k in range(len(probs))]
    for p, fl, g in zip(probs, fields, got):
        with lbm.Lattice(p, prec) as lat:
            lat.init(*fl).step(60)
            want = lat.get_f().cpu().numpy()
        assert np.isfinite(want).all() and np.array_equal(g, want), (p.nx, p.sides)
