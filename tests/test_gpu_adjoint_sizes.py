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


@pytest.mark.parametrize("prec", ["fp64", "fp32_tdf"])
def test_host_and_device_arguments_of_the_adjoint_calls_mix(prec):
    """Each argument of lbm_adjoint_seed and lbm_feq_vjp on the host or on the
    device, on contexts without a staging buffer: the same bits."""
    import torch
    p = W.uniform(37, 11, (1.0, 0.0, 0.0, 1.0), dx=0.1, sides=MIXED)
    rng = np.random.Generator(np.random.PCG64(5))
    dt = np.float64 if prec == "fp64" else np.float32
    fields = [(1.0 + 0.1 * rng.random((p.ny, p.nx))).astype(dt) for _ in range(4)]
    q = [rng.standard_normal((p.ny, p.nx)).astype(dt) for _ in range(4)]
    dev = lambda a: torch.as_tensor(a, device="cuda")
    host = lambda t: t.cpu().numpy() if isinstance(t, torch.Tensor) else t
    want = None
    for mask in (0, 0x3ff, 1, 2, 0x10, 0x20, 0x40, 0x80, 0x155):
        pick = lambda k, a: a.copy() if mask >> k & 1 else dev(a)
        with lbm.Lattice(p, prec) as lat:
            lat.init(*fields)
            abar = pick(4, np.zeros((9, p.ny, p.nx), dt))
            lbm.lbm_adjoint_seed(lat.ctx, pick(0, q[0]), pick(1, q[1]), pick(2, q[2]), pick(3, q[3]), abar)
        with lbm.Lattice(p, prec) as lat:
            g = [pick(6 + k, np.zeros((p.ny, p.nx), dt)) for k in range(4)]
            lbm.lbm_feq_vjp(lat.ctx, *[pick(k, fields[k]) for k in range(4)], pick(5, host(abar)), *g)
            torch.cuda.synchronize()
            got = [host(abar)] + [host(x) for x in g]
        want = want or got
        assert all(np.array_equal(a, b) for a, b in zip(got, want)) and np.abs(got[1]).max() > 0, hex(mask)
