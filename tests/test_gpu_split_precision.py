"""What the kick of light systems may lose by its FP32 pairs: nothing of the
velocity beyond its own rounding.

The velocity after a step's first half kick (the pre-drift state) against
v + (h/2) a in extended precision, a from all pairs, with the drag of
mx_gas_drag (FP64; the drag's impulse is small against the velocity)."""
import numpy as np
import pytest

import oracle as orc
from paper_2601_16791_gb300 import mx, workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

L = np.longdouble
U = 2.0 ** -53


def half_kick(w, x0=None):
    """(start, mx_accel, mx_gas_drag, velocity after the first half kick)"""
    g = mx.System(w)
    mx.mx_set_defer_window(g.h, 0)
    out = [torch.empty((6, w.n), dtype=torch.float64, device="cuda"),
           torch.empty((3, w.n), dtype=torch.float64, device="cuda"),
           torch.zeros((3, w.nsmall), dtype=torch.float64, device="cuda"),
           torch.empty((6, w.n), dtype=torch.float64, device="cuda")]
    if x0 is not None:
        mx.mx_set_state_device(g.h, torch.as_tensor(x0, dtype=torch.float64, device="cuda").contiguous())
    mx.mx_get_state_device(g.h, out[0])
    mx.mx_accel(g.h, out[1])
    if w.params["gas"]["enabled"]:
        mx.mx_gas_drag(g.h, out[2])
    mx.mx_step(g.h, 1)
    mx.mx_predrift_state(g.h, out[3])
    g.close()
    s, a, d, p = (t.cpu().numpy() for t in out)
    return s, a, d, p[3:]


def gravity(w, x):
    """Acceleration of every body in extended precision."""
    p = orc.make_params(w.params)
    _, mu, rc = orc.init(p, w.nbig, w.nsmall, w.m_big, w.xv_helio)
    nb = w.nbig
    out = np.zeros((3, w.n), L)
    for i in range(nb):
        d = x.astype(L) - x[:, i:i + 1].astype(L)
        s2 = (d * d).sum(0)
        s2[i] = 1
        r = np.full(w.n, rc[i])
        r[:nb] = np.maximum(r[:nb], rc[:nb])
        q = np.clip((np.sqrt(s2) - L(0.1) * r) / (L(0.9) * r), 0, 1)
        f = L(mu[i]) * q * q * q * (q * (6 * q - 15) + 10) / (s2 * np.sqrt(s2))
        f[i] = 0
        out -= f * d
    return out


def embryos(nbig, nsmall):
    return W.semiactive_2000big_200k(seed=3, nbig=nbig, nsmall=nsmall)


def disk(nbig, nsmall, rp=(1.0, 100.0)):
    w = W.gas_4core_100k(seed=5, nbig=nbig, nsmall=nsmall)
    w.m_big *= 1e-3
    rng = np.random.default_rng(2)
    w.rp_km = np.exp(rng.uniform(np.log(rp[0]), np.log(rp[1]), nsmall))
    return w


@pytest.mark.parametrize("w", [embryos(40, 2000), embryos(65, 2000), embryos(301, 2000), disk(4, 4000),
                               disk(50, 2000)], ids=["e40", "e65", "e301", "d4", "d50"])
def test_velocity_is_rounded_as_fp64(w):
    """Bound: the pairs' 1.5e-14 of an impulse of at most 1e-3 of the velocity
    (1.5e-17) beside the last rounding's rms of about 5e-17: 5% more."""
    start, _, drag, got = half_kick(w)
    a = gravity(w, start[:3])
    a[:, w.nbig:] += drag.astype(L)
    want = start[3:].astype(L) + L(0.5 * w.params["dt"]) * a
    size = np.sqrt((want * want).sum(0))

    def rms(v):
        return float(np.sqrt(((((v - want) ** 2).sum(0)) / size ** 2).mean()))

    assert rms(got) <= 1.05 * rms(want.astype(np.float64))


def test_near_pairs_and_disk_gravity_stay_fp64():
    """At rest inside the shell of the one big body, with the disk's gravity:
    the velocity is the impulse.  Bound: the product's rounding and the one of
    each sum in the two calls, 4 U of the magnitudes."""
    w = disk(1, 500)
    w.m_big[:] = 1e-7
    w.params["gas"].update(gamma=1.5, r_in_au=0.5, disk_gravity=True, cd_scale=0.0)
    w.params["dt"] = 0.7
    rng = np.random.default_rng(1)
    x = np.zeros((6, w.n))
    x[:3, 0] = w.xv_helio[:3, 0]
    d = rng.normal(size=(3, w.nsmall))
    rc = np.linalg.norm(x[:3, 0]) * 3.0 * (1e-7 / 3.0) ** (1 / 3)
    x[:3, 1:] = x[:3, :1] + d / np.linalg.norm(d, axis=0) * rc * rng.uniform(0.3, 0.9, w.nsmall)
    _, acc, _, got = half_kick(w, x)
    h2 = 0.5 * w.params["dt"]
    s = np.linalg.norm(x[:3, 1:] - x[:3, :1], axis=0)
    err = np.linalg.norm(got - h2 * acc, axis=0)[1:]
    size = h2 * (W.G * 1e-7 / s ** 2 + np.linalg.norm(acc[:, 1:], axis=0))
    assert (err / size).max() <= 4 * U, (err / size).max() / U


def test_strong_drag_stays_fp64():
    """Drag alone (massless big bodies), from weak to many times the velocity.
    A body whose drag changes its velocity relative to the gas by more than
    2^-6 of it keeps FP64: one rounding of v + h a, a as mx_gas_drag returns it
    (U of each component, and U of a, 1.01 for what is of second order).  The
    others add 45 bits of their impulse."""
    w = disk(4, 4000, rp=(1e-5, 100.0))
    w.m_big[:] = 0.0
    start, _, drag, got = half_kick(w)
    nb = w.nbig
    h2 = 0.5 * w.params["dt"]
    want = start[3:, nb:].astype(L) + L(h2) * drag.astype(L)
    g = w.params["gas"]
    x, y = start[:2, nb:]
    R = np.hypot(x, y)
    c_eta = g["hr_1au"] ** 2 * (g["gamma"] + 0.5 - g["flare"] + 1.5) / (2.0 * g["gamma_c"])
    f = np.sqrt(W.G / R * (1.0 - 2.0 * c_eta * R ** (2.0 * g["flare"]))) / R
    dv = start[3:, nb:] + np.stack([f * y, -f * x, 0.0 * x])
    imp = h2 * np.linalg.norm(drag, axis=0)
    strong = imp > 1.02 * 2.0 ** -6 * np.linalg.norm(dv, axis=0)
    weak = imp < 0.98 * 2.0 ** -6 * np.linalg.norm(dv, axis=0)
    assert strong.sum() > 100 and weak.sum() > 100
    err = np.abs(got[:, nb:] - want).astype(np.float64)
    bound = 1.01 * U * (np.abs(want) + h2 * np.abs(drag)).astype(np.float64)
    assert (err / bound)[:, strong].max() <= 1.0, (err / bound)[:, strong].max()
    bound = bound + 2.8e-14 * imp
    assert (err / bound)[:, weak].max() <= 1.0, (err / bound)[:, weak].max()


@pytest.mark.parametrize("far", [4.0, 40.0, 300.0, 480.0])
def test_accel_with_a_distant_big_body(far):
    """The distant body sets the grid of the positions; planetesimals just
    outside the shells of the embryos near 0.5 AU are where it is coarsest.
    Bound: the separation's 2^-54 by coordinate make 3.5 U of a pair, FP64's
    own pair about 10 U (the close ones), two or three roundings of the sums:
    12 U of the pairs' magnitudes."""
    w = embryos(20, 600)
    nb = w.nbig
    xb = w.xv_helio[:, :nb]
    r = np.linalg.norm(xb[:3], axis=0)
    to = np.full(nb, 0.5)
    to[-1] = far
    xb[:3] *= to / r                    # the same orbits at other sizes
    xb[3:] /= np.sqrt(to / r)
    rng = np.random.default_rng(4)
    p = orc.make_params(w.params)
    _, _, rc = orc.init(p, nb, w.nsmall, w.m_big, w.xv_helio)
    b = rng.integers(nb - 1, size=w.nsmall)
    d = rng.normal(size=(3, w.nsmall))
    w.xv_helio[:3, nb:] = xb[:3, b] + d / np.linalg.norm(d, axis=0) * rc[b] * rng.uniform(1.001, 1.5, w.nsmall)
    start, acc, _, _ = half_kick(w)
    x = start[:3]
    err = np.sqrt(((acc - gravity(w, x)) ** 2).sum(0)).astype(np.float64)
    s2 = ((x[:, :, None] - x[:, None, :nb]) ** 2).sum(0)
    s2[s2 == 0] = np.inf
    size = (W.G * w.m_big / s2).sum(1)
    assert (err / size).max() <= 12 * U, (err / size).max() / U
