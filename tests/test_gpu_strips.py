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


def _launched(run, kernel):
    """CTAs of the launches of `kernel` during run(), as the profiler recorded
    them (its first session of a process may record nothing)."""
    import json
    import tempfile
    import torch
    from torch.profiler import ProfilerActivity, profile
    grids = []
    for _ in range(2):
        if not grids:
            with profile(activities=[ProfilerActivity.CPU, ProfilerActivity.CUDA]) as prof:
                run()
                torch.cuda.synchronize()
            with tempfile.NamedTemporaryFile(suffix=".json") as f:
                prof.export_chrome_trace(f.name)
                events = json.load(open(f.name))["traceEvents"]
            grids = [e["args"]["grid"][0] for e in events if e.get("cat") == "kernel" and kernel in e["name"]]
    return grids


@pytest.mark.parametrize("rows,count", [(4, 256), (4, 12), (2, 40)])
def test_the_launch_shape_reported_is_the_one_launched(rows, count):
    """A full wave, and every smaller grid, half the kernel's own and those
    around the shared-memory kernel's full wave (one segment of 128 columns a
    CTA) among them: get_launch and info give the CTAs launched, never more
    than were asked for, and a full wave no more than there are CTAs' worth of
    work (a column at least to each)."""
    st = (1.0, 0.3, 0.05, 1.0)
    probs = [W.uniform(100 + 7 * k % 300, rows, st, dx=DX, sides=(O, O, P, P)) for k in range(count)]
    fields = [W.initial_fields(p, seed=k, sigma=0.01) for k, p in enumerate(probs)]
    segments = sum((p.nx + 127) // 128 for p in probs)
    with lbm.Batch(probs, "fp32_cons") as b:
        b.init(fields).set_launch(1, 0, 5)
        full = b.get_launch()[1]
        for want in sorted({1, 7, full // 2, min(segments, full), min(304, full), full - 1, full}):
            b.set_launch(1, want, 5)
            npt, grid, block = b.get_launch()
            assert (npt, block) == (1, 5) and 1 <= grid <= want and b.info()[0] == grid
            assert set(_launched(lambda: b.step(5), "k_strip")) == {grid}, want
        with pytest.raises(lbm.LbmError) as ei:
            b.set_launch(1, 10 ** 6, 5)
        assert ei.value.status == lbm.LBM_E_INVAL and b.get_launch() == (npt, grid, block)
        (npt, grid, block), _ = b.autotune(steps=5)
        assert (npt, grid, block) == b.get_launch()
        if block:
            assert grid == b.info()[0] and set(_launched(lambda: b.step(block), "k_strip")) == {grid}
    assert full <= sum(p.nx for p in probs)


@pytest.mark.parametrize("rows,sides,grid,block", [(4, (O, O, P, P), 0, 7), (2, (O, O, P, P), 3, 3),
                                                   (4, (O, O, P, P), 1, 5), (4, (O, O, R, R), 0, 5)])
def test_a_barrier_that_misses_an_arrival_times_out_and_the_batch_recovers(rows, sides, grid, block):
    """Failure made on the host: the grid barrier of a blocking launch
    (columns in registers, rounds drawn by ticket or not; the last case in
    shared memory) never completes.  Its bounded wait runs out (0.2 s here),
    LBM_E_TIMEOUT reaches the caller, and after lbm_batch_init the same batch
    gives each problem's own bits."""
    probs = [W.uniform(nx, rows, (1.0, 0.3, 0.05, 1.0), dx=DX, sides=sides) for nx in WIDTHS]
    fields = [W.initial_fields(p, seed=k, sigma=0.01) for k, p in enumerate(probs)]
    lbm.lbm_batch_set_wait_limit(0.2)
    try:
        with lbm.Batch(probs, "fp32_cons") as b:
            b.init(fields).set_launch(1, grid, block).step(block)
            b.sync()
            for restore in (False, True):
                b.plant_stall(0)
                for _ in range(2):  # the second launch finds the status already set
                    b.step(2 * block)
                    with pytest.raises(lbm.LbmError) as ei:
                        b.sync()
                    assert ei.value.status == lbm.LBM_E_TIMEOUT
                if restore:
                    b.plant_stall(-1)
                b.init(fields).step(3 * block)
                b.sync()
                got = [b.get_f(k).cpu().numpy() for k in range(len(probs))]
                for p, fl, g in zip(probs, fields, got):
                    with lbm.Lattice(p, "fp32_cons") as lat:
                        want = lat.init(*fl).step(3 * block).get_f().cpu().numpy()
                    assert np.array_equal(g, want), p.nx
    finally:
        lbm.lbm_batch_set_wait_limit(2.0)
