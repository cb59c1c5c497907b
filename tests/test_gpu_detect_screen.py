"""The encounter test's first screen (encounter_reach: no pair that the exact
test flags may be lost) against the oracle's test of every pair, on end states
that a step need not connect: fast bodies, long and backward steps, big
displacements, at the edges of the 32-body screen and of the staged chunks.
The flag sets are equal except for pairs within 1e-9 of the threshold, which
random states do not hit."""
import numpy as np
import pytest

import oracle as orc
from paper_2601_16791_gb300 import mx, workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("nbig,nsmall,dt,move,fast", [
    (1, 31, 6.0, 0.0, 1.0), (2, 700, 60.0, 0.0, 1.0), (31, 1000, 6.0, 0.05, 1.0),
    (32, 500, -20.0, 0.1, 3.0), (33, 500, 6.0, 0.5, 1.0), (257, 1500, 6.0, 0.02, 1.0),
    (300, 2000, 1.0, 0.3, 20.0),
])
def test_screen_loses_no_encounter(nbig, nsmall, dt, move, fast):
    w = W.semiactive_2000big_200k(seed=9, nbig=nbig, nsmall=nsmall)
    w.params["dt"] = dt
    g = mx.System(w)
    p = orc.make_params(w.params)
    xv0, mu, rc = orc.init(p, w.nbig, w.nsmall, w.m_big, w.xv_helio)
    rng = np.random.default_rng(4)
    rc = rc * rng.choice([1.0, 5.0], size=rc.shape)   # some wide shells
    xv1, _ = orc.drift(p, xv0, dt)
    xv1 = xv1.copy()
    xv1[:3] += move * rng.normal(size=(3, w.n))
    xv0 = xv0.copy()
    xv0[3:] *= fast
    xv1[3:] *= fast * rng.choice([-1.0, 1.0], size=w.n)
    f_ref, p_ref = orc.detect(p, nbig, xv0, xv1, rc)
    cap = len(p_ref) + 64
    dev = [torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda") for a in (xv0, xv1, rc)]
    flags = torch.zeros(w.n, dtype=torch.uint8, device="cuda")
    pairs = torch.zeros(2 * cap, dtype=torch.int32, device="cuda")
    # the entry that takes the changeover radii from the caller
    lib, n = mx.load(), mx.ctypes.c_int(0)
    code = lib.mx_detect_encounters_noalloc(mx.ctypes.byref(mx.make_params(w.params)), nbig, w.n, dev[2].data_ptr(),
                                            dev[0].data_ptr(), dev[1].data_ptr(), flags.data_ptr(),
                                            pairs.data_ptr(), cap, mx.ctypes.byref(n), None)
    assert code == mx.MX_OK, code
    got = pairs.cpu().numpy()[:2 * n.value].reshape(-1, 2)
    want = p_ref[np.lexsort((p_ref[:, 1], p_ref[:, 0]))].reshape(-1, 2)
    assert np.array_equal(got, want)
    assert np.array_equal(flags.cpu().numpy(), f_ref)
    g.close()
