"""lbm_batch_init from device arrays (one launch for many problems) against
lbm_init of each problem: the same operations, so the same bits."""
import numpy as np
import pytest
import torch

from paper_0706_0405_gb300 import lbm
from paper_0706_0405_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_device_arrays_give_the_level_of_each_problem_initialised_alone():
    """103 problems (two launches), odd and even widths, one to nine rows,
    arrays that start 4 bytes off an 8-byte boundary; stepped, given up on and
    initialised again."""
    P, O, R = W.Side("periodic"), W.Side("outflow"), W.Side("reflect")
    shapes = [(1 + (37 * k) % 131, 1 + k % 9) for k in range(103)]
    probs = [W.uniform(nx, ny, (1.0, 0.2, 0.05, 1.0), sides=((O, R, P, P), (R, O, O, R))[k % 2])
             for k, (nx, ny) in enumerate(shapes)]
    host = [W.initial_fields(p, seed=k, sigma=0.01) for k, p in enumerate(probs)]
    total = sum(p.nx * p.ny for p in probs)
    arrays, at = [[], [], [], []], 1  # one element off
    flat = [torch.zeros(total + 1, dtype=torch.float32, device="cuda") for _ in range(4)]
    for p, h in zip(probs, host):
        n = p.nx * p.ny
        for q in range(4):
            view = flat[q][at:at + n]
            view.copy_(torch.as_tensor(np.asarray(h[q]), dtype=torch.float32).reshape(-1))
            arrays[q].append(view)
        at += n
    with lbm.Batch(probs, "fp32_cons") as b:
        lbm.lbm_batch_init(b.handle, *arrays)
        b.step(3)
        lbm.lbm_batch_init(b.handle, *arrays)
        b.sync()
        start = [b.get_f(k).cpu().numpy() for k in range(len(probs))]
        b.step(2)  # reads the ghost cells
        b.sync()
        got = [b.get_f(k).cpu().numpy() for k in range(len(probs))]
    for k, p in enumerate(probs):
        with lbm.Lattice(p, "fp32_cons") as lat:
            lat.init(*[a[k].reshape(p.ny, p.nx) for a in arrays])
            assert np.array_equal(start[k], lat.get_f().cpu().numpy()), p.name
            lat.step(2)
            assert np.array_equal(got[k], lat.get_f().cpu().numpy()), p.name
