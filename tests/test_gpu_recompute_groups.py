"""mx_adjoint_recompute on runs in which many planetesimals are in the groups
that the mode leaves out: every other body has the bits of the same steps taken
one at a time, those that met nothing and, in mode 2, the big bodies of the
groups that are integrated."""
import numpy as np
import pytest

from paper_2601_16791_gb300 import mx, workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def crowd(w, every, bigs):
    """Every `every`-th planetesimal into the outer shell of one of `bigs`,
    moving with it."""
    rng = np.random.default_rng(5)
    j = np.arange(w.nbig, w.n, every)
    b = rng.choice(bigs, size=j.size)
    d = rng.normal(size=(3, j.size))
    hill = np.linalg.norm(w.xv_helio[:3, b], axis=0) * (w.m_big[b] / 3.0) ** (1 / 3)
    w.xv_helio[:, j] = w.xv_helio[:, b]
    w.xv_helio[:3, j] += d / np.linalg.norm(d, axis=0) * hill * rng.uniform(1.0, 2.0, j.size)


@pytest.mark.parametrize("mode,nbig,nsmall,steps", [(0, 4, 600, 4), (0, 1, 33, 2), (2, 60, 700, 3), (2, 200, 900, 2)])
def test_groups_left_out_change_nothing_else(mode, nbig, nsmall, steps):
    if mode == 0:
        w = W.gas_4core_100k(seed=6, nbig=nbig, nsmall=nsmall)
        crowd(w, 3, np.arange(nbig))
    else:
        w = W.semiactive_2000big_200k(seed=6, nbig=nbig, nsmall=nsmall)
        crowd(w, 3, np.arange(nbig // 2, nbig))
        # two pairs of big bodies inside each other's shells
        for i in (0, 2):
            hill = np.linalg.norm(w.xv_helio[:3, i]) * (w.m_big[i] / 3.0) ** (1 / 3)
            w.xv_helio[:, i + 1] = w.xv_helio[:, i]
            w.xv_helio[2, i + 1] += 1.5 * hill
    g = mx.System(w)
    h, n = g.h, w.n
    dev = lambda *s: torch.zeros(s, dtype=torch.float64, device="cuda")
    start = dev(6, n)
    mx.mx_get_state_device(h, start)
    mx.mx_kick_branches(h, 1, 2 * steps + 2)
    mx.mx_encounter_log(h, None, reset=True)
    mx.mx_step(h, steps)
    ever = torch.zeros(n, dtype=torch.uint8, device="cuda")
    nbb = mx.mx_encounter_log(h, ever, reset=False)
    met = ever.bool()
    met[:nbig] = False
    assert int(met.sum()) >= nsmall // 4
    assert (nbb == 0) if mode == 0 else (nbb >= 2)
    mx.mx_kick_branches(h, 2)
    mx._check(mx.load().mx_adjoint_encounters(h, mode), "mx_adjoint_encounters")
    seg, pre, seg2, pre2 = (dev(steps, 6, n) for _ in range(4))
    mx.mx_set_state_device(h, start)
    mx.mx_set_step_index(h, 0)
    for k in range(steps):
        mx.mx_get_state_device(h, seg[k])
        mx.mx_step(h, 1)
        mx.mx_predrift_state(h, pre[k])
    mx.mx_set_state_device(h, start)
    mx.mx_set_step_index(h, 0)
    mx.mx_adjoint_recompute(h, steps, seg2, pre2)
    assert not torch.equal(seg[..., met], seg2[..., met])   # they were left out
    assert torch.equal(seg[..., ~met], seg2[..., ~met])
    assert torch.equal(pre[..., ~met], pre2[..., ~met])
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
