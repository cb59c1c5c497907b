"""The kick's gravity and drag in FP32 pairs against the FP64 ones of mx_accel, at the same
positions.

With every velocity zero, the pre-drift velocity of a step is (h/2) a, a the
acceleration of the first half kick (the momentum is zero, so nothing jumps).
Bound: a pair's acceleration in FP32 pairs is a chain of about twenty
roundings of 2^-48 and smaller, 20 x 2^-48 = 7e-14, times 1.5 for the power
-3/2 and twice for their spread: 2e-13 of the sum of the pairs' magnitudes.
"""
import numpy as np
import pytest

from paper_2601_16791_gb300 import mx, workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

TOL = 2e-13


def place(w, far, shell):
    """Positions of the workload at rest: every 7th planetesimal moved
    off the positions' grid, every 5th close to a big body."""
    x = w.xv_helio.copy()
    x[3:] = 0.0
    nb = w.nbig
    rng = np.random.default_rng(11)
    if shell:
        for j in range(nb, w.n, 5):
            b = rng.integers(nb)
            d = rng.normal(size=3)
            r = np.linalg.norm(x[:3, b])
            rc = 3.0 * r * (w.m_big[b] / 3.0) ** (1 / 3)
            x[:3, j] = x[:3, b] + d / np.linalg.norm(d) * rc * rng.uniform(0.05, 1.3)
    if far:
        x[:3, nb + 3::7] *= 50.0
    return x


@pytest.mark.parametrize("nbig,nsmall,scale,far,shell", [
    (2, 700, 1.0, True, True),
    (64, 300, 1.0, False, False),      # one sum in FP32 pairs
    (65, 1, 1.0, False, False),        # emptied into FP64 every 32
    (65, 1000, 1.0, True, True),
    (96, 333, 0.01, False, True),
    (256, 500, 1.0, False, True),
    (257, 1023, 1.0, True, False),     # a second, one-body chunk
    (300, 2000, 30.0, False, True),
    (550, 700, 1.0, True, True),
    (70, 200, 3000.0, False, False),   # beyond the grid: FP64 throughout
])
def test_split_kick_against_fp64(nbig, nsmall, scale, far, shell):
    w = W.semiactive_2000big_200k(seed=3, nbig=nbig, nsmall=nsmall)
    w.xv_helio[:3] *= scale            # the disk at another size: orbits and Hill radii follow
    w.xv_helio[3:] /= np.sqrt(scale)
    x = place(w, far, shell)
    w.params["dt"] = 1e-3   # the step itself is not under test: bodies at rest fall together
    g = mx.System(w)
    xd = torch.as_tensor(x, dtype=torch.float64, device="cuda").contiguous()
    mx.mx_set_defer_window(g.h, 0)
    mx.mx_set_state_device(g.h, xd)
    acc = torch.empty((3, w.n), dtype=torch.float64, device="cuda")
    mx.mx_accel(g.h, acc)
    pre = torch.empty((6, w.n), dtype=torch.float64, device="cuda")
    mx.mx_step(g.h, 1)
    mx.mx_predrift_state(g.h, pre)
    g.close()
    want = 0.5 * w.params["dt"] * acc.cpu().numpy()
    got = pre[3:].cpu().numpy()
    # magnitude of the pairs (their changeover weight left out below 1)
    d = x[:3, :, None] - x[:3, None, :nbig]
    s2 = (d * d).sum(0)
    s2[s2 == 0] = np.inf
    size = 0.5 * w.params["dt"] * (W.G * w.m_big / s2).sum(1)
    err = np.linalg.norm(got - want, axis=0) / size
    assert err.max() <= TOL, err.max()
    if scale > 1000:
        assert err.max() <= 4e-16
    else:
        assert err.max() > 0.0     # the split path ran


@pytest.mark.parametrize("nbig,nsmall,gas", [
    (1, 257, {}),                      # a core: the FP64 kick
    (3, 3000, {}),
    (33, 1000, {}),                    # a second run of the pair sum
    (64, 500, dict(cd_mode=1)),
    (65, 500, {}),                     # the pair sum goes through FP64
    (4, 2000, dict(gamma=1.5, flare=0.2, r_c_au=20.0, r_in_au=2.0)),
    (4, 2000, dict(gamma=1.5, r_in_au=0.5, disk_gravity=True)),
])
def test_split_drag_against_fp64(nbig, nsmall, gas):
    """A half kick with drag: v1 - v0 against (h/2) mx_accel.  Bound: two
    roundings of the velocity (3e-16 of it), the pairs' 2e-13, and for the drag
    a chain of about twenty products of FP32 pairs, 20 x 2^-45 = 6e-13: 1e-12.
    Radii from a centimetre to a thousand km reach both sides of Re = 1e5 and
    the values that go back to FP64."""
    w = W.gas_4core_100k(seed=5, nbig=nbig, nsmall=nsmall)
    if nbig > 2:
        w.m_big *= 1e-3        # light big bodies; with cores the kick is FP64
    w.params["gas"].update(gas)
    w.params["dt"] = 1e-2      # small bodies stop within days
    rng = np.random.default_rng(2)
    w.rp_km = np.exp(rng.uniform(np.log(1e-5), np.log(1e3), nsmall))
    g = mx.System(w)
    mx.mx_set_defer_window(g.h, 0)
    start = torch.empty((6, w.n), dtype=torch.float64, device="cuda")
    mx.mx_get_state_device(g.h, start)
    acc = torch.empty((3, w.n), dtype=torch.float64, device="cuda")
    drag = torch.empty((3, nsmall), dtype=torch.float64, device="cuda")
    mx.mx_accel(g.h, acc)
    mx.mx_gas_drag(g.h, drag)
    pre = torch.empty((6, w.n), dtype=torch.float64, device="cuda")
    mx.mx_step(g.h, 1)
    mx.mx_predrift_state(g.h, pre)
    g.close()
    h2 = 0.5 * w.params["dt"]
    v0 = start[3:].cpu().numpy()
    x = start[:3].cpu().numpy()
    err = np.linalg.norm(pre[3:].cpu().numpy() - (v0 + h2 * acc.cpu().numpy()), axis=0)
    d = x[:, :, None] - x[:, None, :nbig]
    s2 = (d * d).sum(0)
    s2[s2 == 0] = np.inf
    bound = 3e-16 * np.linalg.norm(v0, axis=0) + TOL * h2 * (W.G * w.m_big / s2).sum(1)
    bound[nbig:] += 1e-12 * h2 * np.linalg.norm(drag.cpu().numpy(), axis=0)
    assert (err / bound).max() <= 1.0, (err / bound).max()


def test_split_keeps_what_fp32_cannot_hold():
    """Masses below FP32's range keep FP64's accuracy in mx_accel (bound: two
    roundings a pair and one of each partial sum, 65 x 2^-52 of the pairs'
    magnitudes), and a drag without bound is reported, not rounded away."""
    w = W.semiactive_2000big_200k(seed=3, nbig=65, nsmall=300)
    w.m_big *= 1e-24
    g = mx.System(w)
    start = torch.empty((6, w.n), dtype=torch.float64, device="cuda")
    acc = torch.empty((3, w.n), dtype=torch.float64, device="cuda")
    mx.mx_get_state_device(g.h, start)
    mx.mx_accel(g.h, acc)
    g.close()
    x = start[:3].cpu().numpy()
    d = x[:, :, None] - x[:, None, :65]
    s2 = (d * d).sum(0)
    s2[s2 == 0] = np.inf
    f = W.G * w.m_big / (s2 * np.sqrt(s2))
    err = np.linalg.norm(acc.cpu().numpy() + (f * d).sum(2), axis=0)
    assert (err / (W.G * w.m_big / s2).sum(1)).max() <= 65 * 2.0 ** -52
    w = W.gas_4core_100k(seed=5, nbig=4, nsmall=500)
    w.m_big *= 1e-3
    w.rp_km[7] = 0.0
    g = mx.System(w)
    with pytest.raises(mx.MxError) as e:
        g.step(1)
    g.close()
    assert e.value.code == 7   # MX_ERR_NONFINITE


@pytest.mark.parametrize("nbig,nsmall", [(65, 40), (128, 700), (257, 1023), (300, 3000)])
def test_parts_of_a_block_change_no_bit(nbig, nsmall):
    """Tiles of 64, 96 or 128 targets share the big bodies among four or two
    parts of a block, tiles of 256 do not: the same accelerations and states."""
    w = W.semiactive_2000big_200k(seed=3, nbig=nbig, nsmall=nsmall)
    out = []
    for tile in (256, 64, 96, 128):
        g = mx.System(w)
        mx.mx_set_tiling(g.h, tile, 0)
        acc = torch.empty((3, w.n), dtype=torch.float64, device="cuda")
        xv = torch.empty((6, w.n), dtype=torch.float64, device="cuda")
        mx.mx_accel(g.h, acc)
        mx.mx_step(g.h, 3)
        mx.mx_get_state_device(g.h, xv)
        out.append((acc.cpu(), xv.cpu()))
        g.close()
    for acc, xv in out[1:]:
        assert torch.equal(acc, out[0][0]) and torch.equal(xv, out[0][1])
