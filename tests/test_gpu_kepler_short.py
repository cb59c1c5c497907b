"""The drift of short steps in relative variables (mx_kepler_short.cuh) against
Gauss' f and g in extended precision, at the edges of its range and beyond,
where the general solver takes over.  Bound: the last addition's rounding and
two or three more at the size of the state's change, at most a few tenths of
it: four half units of 2^-53, 4.5e-16 of the norm."""
import numpy as np
import pytest

from paper_2601_16791_gb300 import mx, workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def gauss(xv, mu, h):
    L = np.longdouble
    x, v = xv[:3].astype(L), xv[3:].astype(L)
    r = np.sqrt((x * x).sum(0))
    a = 1 / (2 / r - (v * v).sum(0) / L(mu))
    n = np.sqrt(L(mu) / a) / a
    es, ec = (x * v).sum(0) / np.sqrt(L(mu) * a), 1 - r / a
    D = n * L(h)
    for _ in range(60):
        s, c1 = np.sin(D), 2 * np.sin(D / 2) ** 2
        D = D - (D - ec * s + es * c1 - n * L(h)) / (1 - ec * (1 - c1) + es * s)
    s, c1 = np.sin(D), 2 * np.sin(D / 2) ** 2
    rn = a * (1 - ec * (1 - c1) + es * s)
    f, g = 1 - a / r * c1, L(h) + (s - D) / n
    fd, gd = -np.sqrt(L(mu) * a) * s / (rn * r), 1 - a / rn * c1
    return np.concatenate([f * x + g * v, fd * x + gd * v])


@pytest.mark.parametrize("nh,emax,sign", [
    (1e-6, 0.05, 1), (0.01, 0.3, -1), (0.1, 0.05, 1), (0.17, 0.3, 1), (0.1995, 0.001, 1), (0.345, 0.001, 1),
    (0.348, 0.001, -1), (0.3, 0.1, 1), (0.02, 0.5, 1),
])
@pytest.mark.parametrize("scale", [1e-3, 1.0, 1e4])
def test_short_drift(nh, emax, sign, scale):
    rng = np.random.default_rng(int(nh * 1e6) + 1)
    n = 1003
    a = scale * rng.uniform(1.0, 1.2, n)
    h = sign * nh * np.sqrt(scale ** 3 / W.G)
    ang = rng.uniform(0, 2 * np.pi, (3, n))
    xv = W.elements_to_xv(W.G, a, rng.uniform(0, emax, n), rng.uniform(0, 0.1, n), *ang)
    w = W.plain_2big_1k()
    w = W.plain_2big_1k(nsmall=n - w.nbig) if w.n != n else w
    g = mx.System(w)
    assert g.n == n
    d = torch.as_tensor(xv, dtype=torch.float64, device="cuda").contiguous()
    mx.mx_kepler_drift(g.h, d, h)
    got = d.cpu().numpy()
    back = torch.as_tensor(xv, dtype=torch.float64, device="cuda").contiguous()
    mx.mx_kepler_drift(g.h, back, 0.0)
    assert np.array_equal(back.cpu().numpy(), xv)
    g.close()
    want = gauss(xv, W.G, h)
    for k in (0, 3):
        err = np.sqrt(((got[k:k + 3] - want[k:k + 3]) ** 2).sum(0) / (want[k:k + 3] ** 2).sum(0))
        assert float(err.max()) <= 4.5e-16, (k, float(err.max()))
