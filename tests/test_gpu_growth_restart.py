"""mx_set_growth on a system that has not stepped: whatever was set before it
(the step index of a restart, a tiling, the recording of the k branches) holds
after it, with an autotune cache that has no entry for the system, so that the
tiling is chosen by trials."""
import numpy as np
import pytest

from paper_2601_16791_gb300 import mx, workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.fixture
def light(tmp_path, monkeypatch):
    """A light growing system's workload and the system without its tracks."""
    monkeypatch.setenv("MX_AUTOTUNE", "1")
    monkeypatch.setenv("MX_AUTOTUNE_CACHE", str(tmp_path / "none.json"))
    w = W.growth_2giant(nsmall=3000, tau_c_days=400.0, tau_g_days=200.0)
    growth, w.growth = w.growth, None
    return w, mx.System(w), lambda s: mx.mx_set_growth(s.h, 0, growth, w.nbig, w.gap_c)


@pytest.mark.parametrize("how", ["state", "index"])
def test_step_index_holds(light, how):
    w, s, grow = light

    def restart(s):
        if how == "state":
            s.set_state(w.xv_helio, mx.MX_COORD_HELIO, 55)
        else:
            mx.mx_set_step_index(s.h, 55)

    out = []
    for calls in ((restart, grow), (grow, restart)):   # the trials are the first one's
        for c in calls:
            c(s)
        radii = mx.mx_planets(s.h, w.nbig)[1]
        s.step(2)
        m, r = mx.mx_planets(s.h, w.nbig)
        out.append((radii, m, r, s.state(mx.MX_COORD_DH)))
        s.close()
        s = mx.System(w)
    s.close()
    assert out[1][1][0] > 10 * W.M_EARTH       # 56 steps of the track, not one
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("tile", [96, 256])
def test_tiling_holds(light, tile):
    w, s, grow = light
    mx.mx_set_tiling(s.h, tile, 0)
    grow(s)
    assert mx.mx_tiling(s.h) == (tile, 0)
    s.close()


def test_recording_starts_empty(light):
    """Recorded on bodies whose Re (below 1e5 after the state is replaced) was
    above 1e5 when the tracks were set: the replay takes the same branches."""
    w, s, grow = light
    mx.mx_kick_branches(s.h, 1, 8)
    grow(s)
    xv = w.xv_helio.copy()
    xv[:3] *= 30.0
    xv[3:] /= np.sqrt(30.0)
    out = []
    for mode in (1, 2):
        if mode == 2:
            mx.mx_kick_branches(s.h, 2)
        s.set_state(xv, mx.MX_COORD_HELIO, 0)
        s.step(1)
        out.append(s.state(mx.MX_COORD_DH))
    s.close()
    assert np.array_equal(*out)
