"""mx_adjoint_recompute against the same steps taken one at a time (mx_step(1)
from each state, mx_predrift_state): the same bits for every body of the groups
the mode integrates and every body that met nothing, and the same cotangents
when the others' are zero (a planetesimal is massless: nothing else reads it)."""
import pytest

from paper_2601_16791_gb300 import mx, workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def dev(*shape):
    return torch.zeros(shape, dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("family,nbig,nsmall,steps,mode", [
    ("gas", 4, 3001, 5, 0), ("gas", 4, 3001, 5, 1), ("gas", 1, 33, 1, 0),
    ("embryos", 400, 1500, 2, 1), ("embryos", 400, 1500, 2, 2), ("embryos", 65, 1, 3, 0),
])
def test_recompute(family, nbig, nsmall, steps, mode):
    w = (W.gas_4core_100k(seed=6, nbig=nbig, nsmall=nsmall) if family == "gas"
         else W.semiactive_2000big_200k(seed=6, nbig=nbig, nsmall=nsmall))
    g = mx.System(w)
    h, n = g.h, w.n
    start = dev(6, n)
    mx.mx_get_state_device(h, start)
    mx.mx_kick_branches(h, 1, 2 * steps + 2)
    mx.mx_encounter_log(h, None, reset=True)
    mx.mx_step(h, steps)
    ever = torch.zeros(n, dtype=torch.uint8, device="cuda")
    nbb = mx.mx_encounter_log(h, ever, reset=False)
    if mode == 0 and nbb:
        pytest.skip("big bodies met: mode 0 is not for this run")
    mx.mx_kick_branches(h, 2)
    mx._check(mx.load().mx_adjoint_encounters(h, mode), "mx_adjoint_encounters")
    met = ever.bool()
    met[:nbig] = False               # every mode follows the big bodies
    seg, pre = dev(steps, 6, n), dev(steps, 6, n)
    mx.mx_set_state_device(h, start)
    mx.mx_set_step_index(h, 0)
    for k in range(steps):
        mx.mx_get_state_device(h, seg[k])
        mx.mx_step(h, 1)
        mx.mx_predrift_state(h, pre[k])
    seg2, pre2 = dev(steps, 6, n), dev(steps, 6, n)
    mx.mx_set_state_device(h, start)
    mx.mx_set_step_index(h, 0)
    mx.mx_adjoint_recompute(h, steps, seg2, pre2)
    same = torch.ones(n, dtype=torch.bool, device="cuda") if mode == 1 else ~met
    assert torch.equal(seg[..., same], seg2[..., same])
    assert torch.equal(pre[..., same], pre2[..., same])
    log = torch.zeros(n, dtype=torch.uint8, device="cuda")
    mx.mx_encounter_log(h, log, reset=False)
    assert torch.equal(log, ever)
    lam0 = torch.randn((6, n), generator=torch.Generator().manual_seed(1), dtype=torch.float64).cuda()
    lam0[:, met] = 0.0
    out = []
    for s, p in ((seg, pre), (seg2, pre2)):
        lam, par = lam0.clone(), dev(3)
        for k in reversed(range(steps)):
            mx.mx_adjoint_step_predrift(h, s[k], p[k], k, lam, par)
        out.append((lam, par))
    g.close()
    assert torch.equal(out[0][0], out[1][0])
    assert torch.equal(out[0][1], out[1][1])
