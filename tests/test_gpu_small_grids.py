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


@pytest.mark.parametrize("prec", ["fp64", "fp32_cons", "fp32_tdf"])
@pytest.mark.parametrize("nx,ny", [(1, 1), (3, 2), (511, 3), (512, 2), (514, 3), (1027, 5)])
def test_read_out_at_the_edges_of_its_vectors_and_units(nx, ny, prec):
    """set_f / get_f keep every value, moments and totals match FP64 sums of
    the stored f, for widths around the 2- and 4-value accesses and the
    512-column units of the totals, in dense arrays of every alignment: the
    totals to 1e-14 of the sum of their terms' magnitudes (a few FP64
    roundings; the FP32 accumulators carry more than 53 bits)."""
    import torch
    p, fields = _problem(nx, ny, WALLS)
    dt = torch.float64 if prec == "fp64" else torch.float32
    rng = np.random.Generator(np.random.PCG64(nx + ny))
    f = torch.tensor(rng.standard_normal((9, ny, nx)) ** 3 + 30.0, dtype=dt, device="cuda")
    with lbm.Lattice(p, prec) as lat:
        for shift in (0, 1):  # a dense array that starts on and off a 16-byte boundary
            buf = torch.empty(f.numel() + shift, dtype=dt, device="cuda")[shift:].view(f.shape)
            buf.copy_(f)
            lbm.lbm_set_f(lat.ctx, buf, 3)
            buf.zero_()
            lbm.lbm_get_f(lat.ctx, buf)
            torch.cuda.synchronize()
            assert torch.equal(buf, f)
        sums = lat.conservation()
        mom = [torch.empty(ny * nx + 1, dtype=dt, device="cuda")[1:] for _ in range(4)]
        lbm.lbm_moments(lat.ctx, *mom)
        torch.cuda.synchronize()
        aligned = lat.moments()
    for a, b in zip(aligned, mom):
        assert torch.equal(a.reshape(-1), b)
    v = f.double().cpu().numpy().reshape(9, -1)
    vx, vy = oracle.velocities(p.c1, p.c2)
    e = vx ** 2 + vy ** 2
    e[0] = p.eta0 ** 2
    for got, w in zip(sums, (np.ones(9), vx, vy, e)):
        terms = (w[:, None] * v).astype(np.longdouble)
        assert abs(got - float(terms.sum())) <= 1e-14 * float(np.abs(terms).sum())


def test_fp32_totals_of_values_whose_sum_leaves_the_fp32_range():
    import torch
    p, _ = _problem(600, 4, PERIODIC)
    with lbm.Lattice(p, "fp32") as lat:
        lat.set_f(torch.full((9, 4, 600), 3e37, dtype=torch.float32, device="cuda"))
        big = lat.conservation()[0]
        f = torch.ones((9, 4, 600), dtype=torch.float32, device="cuda")
        f[2, 1, 7] = float("inf")
        lat.set_f(f)
        assert np.isinf(lat.conservation()[0])
    assert big == pytest.approx(9 * 2400 * float(np.float32(3e37)), rel=1e-14)


# widths and heights around the resident kernel's tiles: one CTA, a last
# narrower tile, a last tile of one column or row, several rounds per CTA, the
# largest grids it takes (their shared memory nearly full) and the first it
# leaves to the one-step kernels
RESIDENT = [(1, 1), (33, 4), (97, 5), (153, 153), (305, 2), (700, 30), (1111, 211), (1240, 310), (1500, 320)]


@pytest.mark.parametrize("prec", ["fp32", "fp32_t64", "fp32_tdf", "fp32_cons"])
@pytest.mark.parametrize("sides", [PERIODIC, WALLS, INFLOW])
@pytest.mark.parametrize("nx,ny", RESIDENT)
def test_steps_in_one_launch_equal_a_launch_a_step(nx, ny, sides, prec):
    """One lbm_step(n) call (several steps per launch where the grid is small
    enough) leaves the bits of n calls of one step, in both level buffers'
    worth of state: after an even and an odd number of steps, after a second
    call on the same context, and with checkpoints recorded on the way."""
    import torch
    p, fields = _problem(nx, ny, sides)
    with lbm.Lattice(p, prec) as one, lbm.Lattice(p, prec) as many:
        one.init(*fields), many.init(*fields)
        lbm.lbm_record(many.ctx, 5)
        for n in (3, 4, 11):
            for _ in range(n):
                one.step(1)
            many.step(n)
            assert torch.equal(one.get_f(), many.get_f()), n
        assert one.health() == many.health()


@pytest.mark.parametrize("sides", [PERIODIC, WALLS, INFLOW])
@pytest.mark.parametrize("nx,ny", [(1, 1), (33, 4), (8, 4), (97, 5), (305, 2), (120, 80), (153, 95), (160, 100)])
def test_fp64_steps_in_one_launch_equal_a_launch_a_step(nx, ny, sides):
    """The FP64 kernel that gives four warps to 32 nodes (one, two and three
    groups a CTA, ragged last groups) does the one-step kernel's operations."""
    import torch
    p, fields = _problem(nx, ny, sides)
    with lbm.Lattice(p, "fp64") as one, lbm.Lattice(p, "fp64") as many:
        one.init(*fields), many.init(*fields)
        for n in (3, 8):
            for _ in range(n):
                one.step(1)
            many.step(n)
            assert torch.equal(one.get_f(), many.get_f()), n


def test_steps_in_one_launch_with_a_moving_split():
    """The double Mach reflection's top boundary moves by whole cells within
    one launch."""
    import torch
    p = W.dmr(40)
    p = p.with_(sides=p.sides[:3] + (Side("dirichlet", "dirichlet", 1.0, 60.0, p.sides[3].state_lo,
                                          p.sides[3].state_hi),))
    assert 60.0 * p.dt * 300 > 20 * p.dx
    with lbm.Lattice(p, "fp32_tdf") as one, lbm.Lattice(p, "fp32_tdf") as many:
        one.init(*W.initial_fields(p)), many.init(*W.initial_fields(p))
        for _ in range(300):
            one.step(1)
        many.step(300)
        assert torch.equal(one.get_f(), many.get_f())


def test_a_captured_call_of_several_steps_replays():
    """lbm_step captured into a CUDA graph: each replay continues from the
    levels the last one left (an even number of steps, so the current level's
    buffer stays the same)."""
    import torch
    p, fields = _problem(200, 12, WALLS)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        lat = lbm.Lattice(p, "fp32_cons").init(*fields)
        lat.step(4)
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            lat.step(6)
        for _ in range(3):
            g.replay()
        s.synchronize()
        got = lat.get_f()
    with lbm.Lattice(p, "fp32_cons") as ref:
        assert torch.equal(ref.init(*fields).step(22).get_f(), got)
    lat.close()


@pytest.mark.parametrize("nx,ny,prec", [(nx, ny, prec) for nx, ny in RESIDENT[:-1]
                                        for prec in ("fp32", "fp32_t64", "fp32_tdf", "fp32_cons")] +
                         [(nx, ny, "fp64") for nx, ny in [(1, 1), (33, 4), (8, 4), (97, 5), (305, 2), (120, 80)]])
def test_small_grids_take_one_launch_for_several_steps(nx, ny, prec):
    """The grids above whose steps are compared do take that launch, from the
    stated number of steps on and with the default launch shape only."""
    p, fields = _problem(nx, ny, INFLOW)
    with lbm.Lattice(p, prec) as lat:
        count = lambda: lbm.lbm_resident_info(lat.ctx)[4]
        lat.init(*fields)
        ctas, depth, steps, levels, n = lbm.lbm_resident_info(lat.ctx)
        assert ctas > 0 and 1 <= depth <= 4 and 3 <= steps <= 30 and levels >= 3 and n == 0
        assert [lat.step(n) and count() for n in (1, 2, steps - 1, steps, 2 * steps)] == [0, 0, 0, 1, 2]
        lbm.lbm_record(lat.ctx, steps)
        lat.step(2 * steps + steps - 1)  # as many to each recorded level, and the others
        assert count() == 4
        lbm.lbm_resident_set(lat.ctx, 3)
        assert [lat.init(*fields).step(n) and count() for n in (2, 3, 11)] == [4, 5, 6]
        lbm.lbm_resident_set(lat.ctx, 0)
        assert lbm.lbm_resident_info(lat.ctx)[2:4] == (steps, levels)
        for bad in (-1, 1, 2):
            with pytest.raises(lbm.LbmError) as ei:
                lbm.lbm_resident_set(lat.ctx, bad)
            assert ei.value.status == lbm.LBM_E_INVAL
        lbm.lbm_set_launch(lat.ctx, 0, 0, 0, 1)
        lat.step(50)
        assert count() == 6
        lat.sync()


@pytest.mark.parametrize("prec", ["fp32", "fp32_t64", "fp32_tdf", "fp32_cons", "fp64"])
@pytest.mark.parametrize("sides", [PERIODIC, WALLS, INFLOW])
@pytest.mark.parametrize("nx,ny", RESIDENT[:-1])
def test_one_launch_from_three_steps_on_equals_a_launch_a_step(nx, ny, sides, prec):
    """As above with that launch from the fewest steps on that the kernel
    takes, also where a launch a step is the default for so few: for the
    lengths around the steps between exchanges, and to recorded levels."""
    import torch
    p, fields = _problem(nx, ny, sides)
    with lbm.Lattice(p, prec) as one, lbm.Lattice(p, prec) as many:
        if lbm.lbm_resident_info(many.ctx)[0] == 0:
            assert prec == "fp64" and nx * ny > 9000
            return
        lbm.lbm_resident_set(many.ctx, 3)
        one.init(*fields), many.init(*fields)
        for n in (3, 4, 5, 6, 20):
            if n == 20:
                lbm.lbm_record(many.ctx, 7)
            for _ in range(n):
                one.step(1)
            many.step(n)
            assert torch.equal(one.get_f(), many.get_f()), n
        assert lbm.lbm_resident_info(many.ctx)[4] == 7 and lbm.lbm_resident_info(one.ctx)[4] == 0
        assert one.health() == many.health()


def test_larger_grids_take_a_launch_a_step():
    p, fields = _problem(*RESIDENT[-1], WALLS)
    with lbm.Lattice(p, "fp32") as lat:
        lat.init(*fields).step(5).sync()
        assert lbm.lbm_resident_info(lat.ctx) == (0, 0, 0, 0, 0)
        for call in (lambda: lbm.lbm_plant_stall(lat.ctx, True), lambda: lbm.lbm_resident_set(lat.ctx, 3)):
            with pytest.raises(lbm.LbmError) as ei:
                call()
            assert ei.value.status == lbm.LBM_E_STATE


@pytest.mark.parametrize("nx,ny,prec", [(2000, 4, "fp32_tdf"), (400, 100, "fp32_cons"), (400, 4, "fp64"),
                                        (120, 80, "fp64"), (1240, 310, "fp32_t64")])
def test_a_value_that_never_arrives_times_out_and_the_context_recovers(nx, ny, prec):
    """Failure made on the host: the launches lack a CTA, so that those next
    to it wait for values that nobody publishes.  Their bounded waits run out
    (0.2 s here), all CTAs leave, LBM_E_TIMEOUT reaches the caller and stays
    until lbm_init, after which the same context gives the bits of one that
    never failed."""
    import torch
    p, fields = _problem(nx, ny, WALLS)
    lbm.lbm_batch_set_wait_limit(0.2)
    try:
        with lbm.Lattice(p, prec) as lat, lbm.Lattice(p, prec) as ref:
            lbm.lbm_resident_set(lat.ctx, 3)
            for first in (3, 4, 7):  # the exchange buffer's halves in either order
                lat.init(*fields).step(first)
                lat.sync()
                lbm.lbm_plant_stall(lat.ctx, True)
                for n in (9, 4):  # the second launch finds the status already set
                    lat.step(n)
                    with pytest.raises(lbm.LbmError) as ei:
                        lat.sync()
                    assert ei.value.status == lbm.LBM_E_TIMEOUT
                lbm.lbm_plant_stall(lat.ctx, False)
            got = lat.init(*fields).step(25).get_f()
            lat.sync()
            assert torch.equal(ref.init(*fields).step(25).get_f(), got)
    finally:
        lbm.lbm_batch_set_wait_limit(2.0)


def test_contexts_on_several_streams_at_once():
    """Launches of several steps queued from one thread per context, each on a
    stream of its own, beside other work on the device: the bits of each
    context stepped alone."""
    import threading
    import torch
    cases = [(2000, 4, "fp32_tdf"), (900, 300, "fp32_cons"), (400, 100, "fp32"), (400, 4, "fp64"),
             (1024, 256, "fp32_t64"), (120, 80, "fp64")]
    problems = [_problem(nx, ny, WALLS) for nx, ny, _ in cases]
    want = []
    for (p, fields), (_, _, prec) in zip(problems, cases):
        with lbm.Lattice(p, prec) as lat:
            want.append(lat.init(*fields).step(300).get_f())
    got = [None] * len(cases)

    def run(k):
        with torch.cuda.stream(torch.cuda.Stream()):
            with lbm.Lattice(problems[k][0], cases[k][2]) as lat:
                lat.init(*problems[k][1])
                for _ in range(10):
                    lat.step(30)
                lat.sync()
                got[k] = lat.get_f()

    a = torch.ones((4096, 4096), device="cuda")
    for _ in range(20):
        a = a * 0.5 + 1.0
    threads = [threading.Thread(target=run, args=(k,)) for k in range(len(cases))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for w, g in zip(want, got):
        assert g is not None and torch.equal(w, g)


@pytest.mark.parametrize("nx,ny,prec", [(256, 8, "fp64"), (400, 100, "fp32_tdf")])
def test_a_recomputation_that_gives_up_is_reported_by_the_adjoint(nx, ny, prec):
    """The forward steps run through; the levels between the checkpoints are
    recomputed by launches that lack a CTA.  lbm_adjoint_step returns
    LBM_E_TIMEOUT and leaves the tau derivative alone; after lbm_init the same
    context gives the gradient of one that never failed."""
    import ctypes
    import torch
    p, fields = _problem(nx, ny, WALLS)

    def gradient(lat, stall):
        lat.init(*fields)
        lbm.lbm_record(lat.ctx, 10)
        lat.step(20).sync()
        abar = torch.ones((9, ny, nx), dtype=lat.dtype, device="cuda")
        dtau = ctypes.c_double(7.0)
        if stall:
            lbm.lbm_plant_stall(lat.ctx, True)
        st = lbm.load().lbm_adjoint_step(lat.ctx, 20, ctypes.c_void_p(abar.data_ptr()), ctypes.byref(dtau))
        lbm.load().lbm_plant_stall(lat.ctx, 0)
        return st, dtau.value, abar

    lbm.lbm_batch_set_wait_limit(0.2)
    try:
        with lbm.Lattice(p, prec) as lat, lbm.Lattice(p, prec) as ref:
            lbm.lbm_resident_set(lat.ctx, 3), lbm.lbm_resident_set(ref.ctx, 3)
            assert gradient(lat, True)[:2] == (lbm.LBM_E_TIMEOUT, 7.0)
            got, want = gradient(lat, False), gradient(ref, False)
    finally:
        lbm.lbm_batch_set_wait_limit(2.0)
    assert got[0] == want[0] == lbm.LBM_OK and got[1] == want[1] != 7.0 and torch.equal(got[2], want[2])


# Narrow grids (units of several rows, runs in the order of the rows), widths on
# either side of where rows are cut into patches, and large grids whose rows
# allow 16-byte, 8-byte or single accesses
READ_OUT = [(1, 130), (2, 257), (3, 1000), (4, 129), (5, 64), (7, 33), (16, 100), (17, 9), (63, 130), (64, 65),
            (65, 40), (100, 5), (129, 900), (257, 5), (1, 40000), (3, 70001), (1024, 1025), (1030, 1031), (1027, 1029)]


@pytest.mark.parametrize("prec", ["fp64", "fp32_cons", "fp32_t64"])
@pytest.mark.parametrize("nx,ny", READ_OUT)
def test_read_out_of_narrow_and_large_grids(nx, ny, prec):
    """Initial levels and moments are those of the same nodes in one row, on
    and off 16-byte boundaries; the ghost cells of an initial level are those
    that lbm_set_f makes (one step from either); totals to 1e-14 of the sum of
    their terms' magnitudes, also where a sum is taken again in FP64."""
    import torch
    p, fields = _problem(nx, ny, WALLS)
    row, _ = _problem(nx * ny, 1, WALLS)
    dt = torch.float64 if prec == "fp64" else torch.float32
    shifted = []
    for a in fields:
        buf = torch.empty(nx * ny + 1, dtype=dt, device="cuda")[1:]
        buf.copy_(torch.as_tensor(a.reshape(-1)))
        shifted.append(buf)
    with lbm.Lattice(p, prec) as lat, lbm.Lattice(row.with_(tau=p.tau, dt=p.dt), prec) as line:
        f = lat.init(*fields).get_f()
        assert torch.equal(line.init(*[a.reshape(1, -1) for a in fields]).get_f().reshape(9, -1), f.reshape(9, -1))
        for a, b in zip(lat.moments(), line.moments()):
            assert torch.equal(a.reshape(-1), b.reshape(-1))
        sums = lat.conservation()
        after = lat.step(1).get_f()
        lbm.lbm_init(lat.ctx, *shifted)
        assert torch.equal(lat.get_f(), f)
        assert torch.equal(lat.set_f(f).step(1).get_f(), after)
        if prec != "fp64":
            g = f.clone()
            g[3, ny - 1, nx - 1] = 3e38
            g[3, 0, 0] = 3e38
            big = lat.set_f(g).conservation()[0]
            want = g.double().sum(dtype=torch.float64).item()
            assert np.isfinite(big) and abs(big - want) <= 1e-14 * want
    v = f.double().cpu().numpy().reshape(9, -1)
    vx, vy = oracle.velocities(p.c1, p.c2)
    e = vx ** 2 + vy ** 2
    e[0] = p.eta0 ** 2
    for got, w in zip(sums, (np.ones(9), vx, vy, e)):
        terms = (w[:, None] * v).astype(np.longdouble)
        assert abs(got - float(terms.sum())) <= 1e-14 * float(np.abs(terms).sum())
