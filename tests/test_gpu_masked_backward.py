"""A masked backward leaves out the encounter groups it does not differentiate.
The state that it leaves in the system is the run's own all the same."""
import numpy as np
import pytest

from paper_2601_16791_gb300 import autograd, mx, workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("nsteps,every", [(4, 2), (5, 2), (3, 3), (2, 7)])
def test_backward_leaves_the_runs_state(nsteps, every):
    w = W.gas_4core_100k(seed=6, nsmall=600)
    nb = w.nbig
    # a third of the planetesimals inside the cores' changeover shells, moving
    # with them: encounters from the first step on
    rng = np.random.default_rng(3)
    for j in range(nb, w.n, 3):
        b = rng.integers(nb)
        r = np.linalg.norm(w.xv_helio[:3, b])
        d = rng.normal(size=3)
        w.xv_helio[:, j] = w.xv_helio[:, b]
        w.xv_helio[:3, j] += d / np.linalg.norm(d) * r * (w.m_big[b] / 3.0) ** (1 / 3) * rng.uniform(0.5, 2.0)
    traj = autograd.Trajectory(w)
    xv = torch.from_numpy(w.xv_helio).cuda().requires_grad_(True)
    g = w.params["gas"]
    gas = torch.tensor([g["sigma1_gcm2"], g["gamma"], g["cd_scale"]], dtype=torch.float64, device="cuda")
    weight = torch.ones(w.n, dtype=torch.float64, device="cuda")
    autograd.semimajor_loss(traj, xv, gas, weight, nsteps, every, True).backward()
    left = torch.empty((6, w.n), dtype=torch.float64, device="cuda")
    mx.mx_get_state_device(traj.h, left)
    _, step = mx.mx_get_state(traj.h, w.n)
    # the same run again, as far as that step
    _, ever, _ = traj.run(xv, gas, min(every, nsteps), every)
    again = torch.empty_like(left)
    mx.mx_get_state_device(traj.h, again)
    traj.close()
    assert int(ever[nb:].sum()) > 50
    assert step == min(every, nsteps)
    assert torch.equal(left, again)
