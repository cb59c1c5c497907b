"""The encounter pairs of mx_detect_encounters in order at every size of the key
sort: ranked by all SMs up to 16,384 keys, sorted by one block beyond, and cut
at the system's pair capacity.  The pairs are known: planetesimals at rest
inside the shell of one or two big bodies, the others far from both."""
import numpy as np
import pytest

import oracle as orc
from paper_2601_16791_gb300 import mx, workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def meet(npairs, pair_cap):
    """(status, count, pairs, flags) and the pairs and flags expected"""
    nbig, nsmall = 3, max(64, npairs + 40)
    w = W.semiactive_2000big_200k(seed=4, nbig=nbig, nsmall=nsmall)
    w.params["pair_cap"] = pair_cap
    p = orc.make_params(w.params)
    xv, _, rc = orc.init(p, nbig, nsmall, w.m_big, w.xv_helio)
    rng = np.random.default_rng(npairs)
    host = np.full(nsmall, -1)
    met = rng.permutation(nsmall)[:npairs]
    host[met] = rng.integers(2, size=npairs)
    x = np.zeros((6, w.n))
    x[0, :nbig] = [1.0, 2.0, 3.0]
    d = rng.normal(size=(3, nsmall))
    d /= np.linalg.norm(d, axis=0)
    x[:3, nbig:] = np.where(host < 0, 20.0 * d, x[:3, host] + 0.5 * rc[host] * d)
    j = np.flatnonzero(host >= 0)
    want = np.stack([host[j], nbig + j], axis=1)
    want = want[np.lexsort((want[:, 1], want[:, 0]))]
    flags = np.zeros(w.n, np.uint8)
    flags[want.ravel()] = 1
    g = mx.System(w)
    t = torch.as_tensor(x, device="cuda")
    out = torch.zeros(w.n, dtype=torch.uint8, device="cuda")
    pairs = torch.full((npairs + 8, 2), -1, dtype=torch.int32, device="cuda")
    n = mx.ctypes.c_int(0)
    code = mx.load().mx_detect_encounters(g.h, t.data_ptr(), t.data_ptr(), out.data_ptr(),
                                          pairs.data_ptr(), npairs + 8, mx.ctypes.byref(n))
    g.close()
    return code, n.value, pairs.cpu().numpy(), out.cpu().numpy(), want, flags


@pytest.mark.parametrize("npairs", [0, 1, 7, 9, 4097, 16383, 16384, 16385, 40000])
def test_pairs_come_in_order(npairs):
    code, n, pairs, flags, want, fref = meet(npairs, 1 << 16)
    assert code == mx.MX_OK
    assert n == npairs
    assert np.array_equal(pairs[:npairs], want)
    assert (pairs[npairs:] == -1).all()
    assert np.array_equal(flags, fref)


@pytest.mark.parametrize("npairs,cap", [(1001, 1000), (16385, 16384), (20000, 17000)])
def test_more_pairs_than_the_system_holds(npairs, cap):
    """Refused; the pairs it kept are true ones, each once, in order."""
    code, n, pairs, _, want, _ = meet(npairs, cap)
    assert code == 6   # MX_ERR_PAIR_OVERFLOW
    assert n == npairs
    got = [tuple(q) for q in pairs[:cap]]
    assert got == sorted(set(got))
    assert set(got) <= {tuple(q) for q in want}
