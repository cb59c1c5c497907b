"""The calls this framework is used for, as cases that can be timed and compared.

A case names a kind of call, the shape of the system it is made on and the
steps of one pass.  Shapes and distributions are those of the package's
workloads (paper_2601_16791_gb300/workloads.py): planets among massless
planetesimals, gas disks with growing cores, self-gravitating embryo disks and
ensembles of disks of uneven size.

Kinds:
  step      restart from a checkpoint on the device, advance, read the state:
            the loop of a simulation (a pass starts from the same state, so
            that it can be repeated)
  io        the state from pinned host memory, one step, the state back: a
            host program that keeps the bodies itself
  ensemble  the same as step for a batch of independent systems
  adjoint   the differentiable run, forward and backward: loss, gradient of
            the initial state and of the gas parameters
  accel     the kick's acceleration at the current state (diagnostics, other
            integrators)
  drift     the Kepler drift of a buffer of bodies (other splittings)
  detect    the encounter test between two states
"""
import ctypes
import math

import numpy as np
import torch

from paper_2601_16791_gb300 import autograd, mx
from paper_2601_16791_gb300 import workloads as W

DT = {"plain": 8.0, "gas": 10.0, "embryos": 6.0, "growth": 10.0}


def listed():
    return [
        # two giants and a small swarm, a call of fifty short steps: launches and latency
        {"name": "plain_step_1k", "kind": "step", "family": "plain", "nbig": 2, "nsmall": 1000, "steps": 50},
        # growing cores in a gas disk: the paper's main use, in the loop of a long run
        {"name": "gas_step_100k", "kind": "step", "family": "gas", "nbig": 4, "nsmall": 100_000, "steps": 20},
        # the same disk, driven step by step from the host
        {"name": "gas_io_100k", "kind": "io", "family": "gas", "nbig": 4, "nsmall": 100_000, "steps": 1},
        # two forming giants with gaps in the gas
        {"name": "growth_step_24k", "kind": "step", "family": "growth", "nbig": 2, "nsmall": 24_000, "steps": 20},
        # a self-gravitating embryo disk at full size: gravity of 2,000 sources, many encounters
        {"name": "embryos_step_200k", "kind": "step", "family": "embryos", "nbig": 2000, "nsmall": 200_000, "steps": 2},
        # a smaller one of odd sizes, as in a convergence study
        {"name": "embryos_step_20k", "kind": "step", "family": "embryos", "nbig": 301, "nsmall": 20_011, "steps": 4},
        # a parameter study: disks of 2 to 50 big bodies and 1,000 to 200,000 planetesimals in one batch
        {"name": "ensemble_step_64", "kind": "ensemble", "nsys": 64, "most": 200_000, "steps": 3},
        # fitting a gas disk: ten steps forward and back, encounters masked
        {"name": "adjoint_gas_50k", "kind": "adjoint", "family": "gas", "nbig": 4, "nsmall": 50_000, "steps": 10, "mask": True},
        # the derivative through every encounter of an embryo disk
        {"name": "adjoint_embryos_20k", "kind": "adjoint", "family": "embryos", "nbig": 1000, "nsmall": 20_000, "steps": 2, "mask": False},
        # single parts at full size
        {"name": "accel_embryos_200k", "kind": "accel", "family": "embryos", "nbig": 2000, "nsmall": 200_000},
        {"name": "drift_200k", "kind": "drift", "n": 200_000},
        {"name": "detect_200k", "kind": "detect", "family": "embryos", "nbig": 2000, "nsmall": 200_000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "io", "ensemble", "adjoint", "accel", "drift", "detect"])
    family = rng.choice(["plain", "gas", "growth", "embryos"])
    if kind == "ensemble":
        return {"kind": kind, "nsys": _log(rng, 4, 64), "most": _log(rng, 5000, 200_000), "steps": rng.randint(2, 3)}
    if kind == "drift":
        return {"kind": kind, "n": _log(rng, 1000, 200_000)}
    if kind == "detect":
        return {"kind": kind, "family": "embryos", "nbig": _log(rng, 100, 2000), "nsmall": _log(rng, 5000, 200_000)}
    if kind == "accel":
        family = rng.choice(["gas", "embryos"])
        return {"kind": kind, "family": family, "nbig": 4 if family == "gas" else _log(rng, 20, 2000),
                "nsmall": _log(rng, 1000, 200_000)}
    if kind == "adjoint":
        family = rng.choice(["gas", "embryos"])
        nbig = rng.randint(2, 8) if family == "gas" else _log(rng, 70, 1000)
        return {"kind": kind, "family": family, "nbig": nbig, "nsmall": _log(rng, 1000, 50_000 if family == "gas" else 20_000),
                "steps": rng.randint(2, 10) if family == "gas" else 2, "mask": rng.random() < 0.5}
    nbig = {"plain": 2, "gas": rng.randint(2, 8), "growth": 2, "embryos": _log(rng, 20, 2000)}[family]
    nsmall = _log(rng, 1000, {"plain": 100_000, "gas": 100_000, "growth": 24_000, "embryos": 200_000}[family])
    if kind == "io":
        return {"kind": kind, "family": family, "nbig": nbig, "nsmall": nsmall, "steps": 1}
    return {"kind": kind, "family": family, "nbig": nbig, "nsmall": nsmall,
            "steps": rng.randint(1, 2) if family == "embryos" else rng.randint(1, 50 if family == "plain" else 20)}


# ------------------------------------------------------------------- inputs
class _Draws:
    """Seeded draws on the GPU (the states of the workloads, made faster)."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda").manual_seed(int(seed))

    def uniform(self, n, lo, hi):
        return lo + (hi - lo) * torch.rand(n, generator=self.g, device="cuda", dtype=torch.float64)

    def rayleigh(self, n, sigma):
        return sigma * torch.sqrt(-2.0 * torch.log1p(-torch.rand(n, generator=self.g, device="cuda", dtype=torch.float64)))

    def log_uniform(self, n, lo, hi):
        return torch.exp(self.uniform(n, math.log(lo), math.log(hi)))

    def bodies(self, gm, a, sigma_e, sigma_i):
        """Heliocentric states [6, n] of bodies on orbits of semimajor axis a."""
        n = a.numel()
        e = self.rayleigh(n, sigma_e).clamp(max=0.9)
        inc = self.rayleigh(n, sigma_i)
        node, peri, M = (self.uniform(n, 0.0, 2 * math.pi) for _ in range(3))
        E = M.clone()
        for _ in range(20):
            E = E - (E - e * torch.sin(E) - M) / (1.0 - e * torch.cos(E))
        cE, sE, rt = torch.cos(E), torch.sin(E), torch.sqrt(1.0 - e * e)
        fac = torch.sqrt(gm / a) / (1.0 - e * cE)
        xo, yo, vxo, vyo = a * (cE - e), a * rt * sE, -fac * sE, fac * rt * cE
        cO, sO, cw, sw = torch.cos(node), torch.sin(node), torch.cos(peri), torch.sin(peri)
        ci, si = torch.cos(inc), torch.sin(inc)
        r = ((cO * cw - sO * sw * ci, -cO * sw - sO * cw * ci),
             (sO * cw + cO * sw * ci, -sO * sw + cO * cw * ci), (sw * si, cw * si))
        return torch.stack([p * xo + q * yo for p, q in r] + [p * vxo + q * vyo for p, q in r])


def _disk(d, family, nbig, nsmall, steps):
    """A workloads.Workload of the family's distributions at these sizes."""
    rp = rho = torch.ones(nsmall, dtype=torch.float64, device="cuda")
    growth = None
    if family == "plain":     # as plain_2big_1k
        m = torch.tensor([W.M_JUP, 0.3 * W.M_JUP], dtype=torch.float64, device="cuda")
        ab, eb, ib = torch.tensor([5.2, 9.5], dtype=torch.float64, device="cuda"), 0.02, 0.008
        amin, amax, es, is_ = 2.0, 12.0, 0.01, 0.005
    elif family == "gas":     # as gas_4core_100k
        m, ab = d.uniform(nbig, 10.0, 30.0) * W.M_EARTH, d.uniform(nbig, 3.0, 10.0)
        eb, ib, amin, amax, es, is_ = 0.01, 0.005, 1.0, 15.0, 0.01, 0.005
    elif family == "growth":  # as growth_2giant, part way through its growth
        m = torch.full((2,), 0.01 * W.M_EARTH, dtype=torch.float64, device="cuda")
        ab = torch.tensor([10.0, 20.0], dtype=torch.float64, device="cuda")
        eb, ib, amin, amax, es, is_ = 0.01, 0.005, 1.0, 25.0, 0.01, 0.005
        growth = dict(m0=m.cpu().numpy(), mc=np.full(2, 15.0 * W.M_EARTH), mf=np.array([300.0, 100.0]) * W.M_EARTH,
                      tau_c=np.full(2, 400.0), tau_g=np.full(2, 200.0), delta_r=np.full(2, 0.01),
                      grows=np.ones(2, dtype=np.int32))
    elif family == "member":  # as one of ensemble_256
        m, ab = d.log_uniform(nbig, W.M_MOON, W.M_MARS), d.uniform(nbig, 1.0, 15.0)
        eb, ib, amin, amax, es, is_ = 0.01, 0.005, 1.0, 15.0, 0.01, 0.005
    else:                     # as semiactive_2000big_200k
        m, ab = d.log_uniform(nbig, W.M_MOON, W.M_MARS), d.uniform(nbig, 0.5, 4.0)
        eb, ib, amin, amax, es, is_ = 0.02, 0.01, 0.5, 4.0, 0.02, 0.01
    gas = family in ("gas", "growth", "member")
    if gas:
        rp, rho = d.log_uniform(nsmall, 1.0, 100.0), d.uniform(nsmall, 1.0, 3.0)
    xv = torch.cat([d.bodies(W.G * (1.0 + m), ab, eb, ib),
                    d.bodies(W.G, d.uniform(nsmall, amin, amax), es, is_)], dim=1)
    sigma1 = 1700.0 * (float(d.uniform(1, 0.3, 3.0)) if family == "member" else 1.0)
    params = W.default_params(DT.get(family, 10.0), W.default_gas(gas, sigma1=sigma1))
    return W.Workload(name=family, params=params, nbig=int(m.numel()), nsmall=int(nsmall), m_big=m.cpu().numpy(),
                      xv_helio=np.ascontiguousarray(xv.cpu().numpy()), rp_km=rp.cpu().numpy(), rhop=rho.cpu().numpy(),
                      nsteps=int(steps), growth=growth)


def _members(seed, nsys, most):
    """(big bodies, planetesimals) of each system of an ensemble: 2 to 50,
    uniform, and 1,000 to `most`, log-uniform, in strata so that ensembles of
    different seeds cost the same."""
    r = np.random.default_rng(12345 + nsys)
    q = (r.permutation(nsys) + 0.5) / nsys
    k = 2 + (r.permutation(nsys) * 49) // nsys
    return [(int(b), int(round(math.exp(math.log(1000) + float(u) * math.log(most / 1000))))) for b, u in zip(k, q)]


def prepare(case, seed):
    d = _Draws(seed)
    kind = case["kind"]
    if kind == "drift":
        xv = d.bodies(W.G, d.uniform(case["n"], 1.0, 15.0), 0.05, 0.02)
        w = _disk(d, "plain", 2, case["n"] - 2, 1)   # the call drifts as many bodies as the system has
        return {"kind": kind, "sys": mx.System(w), "xv": xv.contiguous(), "out": torch.empty_like(xv), "h": 10.0}
    if kind == "ensemble":
        ws = [_disk(d, "member", b, n, case["steps"]) for b, n in _members(seed, case["nsys"], case["most"])]
        s = mx.Batch(ws)
        n = s.n
    else:
        w = _disk(d, case["family"], case["nbig"], case["nsmall"], case.get("steps", 1))
        n = w.n
        if kind == "adjoint":
            weight = torch.zeros(n, dtype=torch.float64, device="cuda")
            weight[w.nbig:] = 1.0 / w.nsmall
            g = w.params["gas"]
            return {"kind": kind, "traj": autograd.Trajectory(w), "w": weight,
                    "xv": torch.from_numpy(w.xv_helio).cuda().requires_grad_(True),
                    "gas": torch.tensor([g["sigma1_gcm2"], g["gamma"], g["cd_scale"]], dtype=torch.float64,
                                        device="cuda", requires_grad=True),
                    "steps": case["steps"], "every": max(1, case["steps"] // 2), "mask": case["mask"]}
        s = mx.System(w)
    state = {"kind": kind, "sys": s, "steps": case.get("steps", 1),
             "out": torch.empty((6, n), dtype=torch.float64, device="cuda")}
    if kind == "io":
        state["in"] = torch.from_numpy(w.xv_helio).clone().pin_memory()
        state["back"] = torch.empty((6, n), dtype=torch.float64).pin_memory()
    elif kind == "accel":
        state["out"] = torch.empty((3, n), dtype=torch.float64, device="cuda")
    elif kind == "detect":
        # a step's end points: the state, and the state drifted over the step
        start = torch.empty((6, n), dtype=torch.float64, device="cuda")
        mx.mx_get_state_device(s.h, start)
        end = start.clone()
        mx.mx_kepler_drift(s.h, end, w.params["dt"])
        state.update(start=start, end=end, cap=1 << 18,
                     flags=torch.empty(n, dtype=torch.uint8, device="cuda"),
                     pairs=torch.zeros((1 << 18, 2), dtype=torch.int32, device="cuda"))
    else:
        state["start"] = torch.empty((6, n), dtype=torch.float64, device="cuda")
        mx.mx_get_state_device(s.h, state["start"])
    return state


# --------------------------------------------------------------------- pass
def run(state):
    kind = state["kind"]
    if kind == "adjoint":
        xv, gas = state["xv"], state["gas"]
        L = autograd.semimajor_loss(state["traj"], xv, gas, state["w"], state["steps"], state["every"], state["mask"])
        grad_xv, grad_gas = torch.autograd.grad(L, (xv, gas))
        return {"loss": L.detach(), "state": grad_xv, "gas": grad_gas}
    h = state["sys"].h
    if kind == "drift":
        state["out"].copy_(state["xv"])
        mx.mx_kepler_drift(h, state["out"], state["h"])
    elif kind == "accel":
        mx.mx_accel(h, state["out"])
    elif kind == "detect":
        n = mx.mx_detect_encounters(h, state["start"], state["end"], state["flags"], state["pairs"], state["cap"])
        return {"count": n, "flags": state["flags"], "pairs": state["pairs"]}   # zeros past the count
    elif kind == "io":
        lib = mx.load()
        step = ctypes.c_longlong(0)
        for code in (lib.mx_set_state(h, state["in"].data_ptr(), mx.MX_COORD_HELIO, 0), lib.mx_step(h, 1),
                     lib.mx_get_state(h, state["back"].data_ptr(), mx.MX_COORD_HELIO, ctypes.byref(step))):
            if code != mx.MX_OK:
                raise mx.MxError(code, "step from the host")
        return state["back"]
    else:
        mx.mx_set_state_device(h, state["start"])
        mx.mx_set_step_index(h, 0)
        mx.mx_step(h, state["steps"])
        mx.mx_get_state_device(h, state["out"])
    return state["out"]


def work(case):
    """Bytes: the state (and drag constants) read once and written once.
    Operations: 20 per (body, big body) pair and half kick pair, 30 per pair
    tested for an encounter, 343 per drift, 2 x 97 per body's drag and kicks;
    an adjoint pass goes forward, recomputes and reverses (twice the pair's
    operations)."""
    kind = case["kind"]
    if kind == "drift":
        return {"bytes": 96 * case["n"], "flops": 343 * case["n"]}
    if kind == "ensemble":
        sizes = _members(0, case["nsys"], case["most"])
        n = sum(b + s for b, s in sizes)
        pairs = sum(b * (b + s) for b, s in sizes)
        return {"bytes": 112 * n, "flops": case["steps"] * (50 * pairs + (343 + 194) * n)}
    n = case["nbig"] + case["nsmall"]
    pairs = case["nbig"] * n
    gas = case["family"] in ("gas", "growth")
    if kind == "accel":
        return {"bytes": (72 + 16 * gas) * n, "flops": 20 * pairs + 88 * gas * n}
    if kind == "detect":
        return {"bytes": 97 * n, "flops": 30 * pairs}
    step = 50 * pairs + (343 + (194 if gas else 18)) * n
    if kind == "adjoint":
        return {"bytes": 152 * n, "flops": case["steps"] * (4 * step)}
    return {"bytes": (96 + 16 * gas) * n, "flops": case["steps"] * step}


# -------------------------------------------------------------------- exact
def exact(case, seed):
    """The parts that have a closed statement, in 64 bits: the kick's
    acceleration (pair sums with the changeover weight; no gas) and the drift.
    A step goes through adaptive Bulirsch-Stoer integrations, which have none
    to better than their tolerance; the encounter test returns whole values."""
    if case["kind"] == "drift":
        s = prepare(case, seed)
        return _kepler(s["xv"], W.G, s["h"])
    if case["kind"] == "accel" and case["family"] == "embryos":
        w = _disk(_Draws(seed), case["family"], case["nbig"], case["nsmall"], 1)
        x = torch.from_numpy(w.xv_helio).cuda()
        m = torch.from_numpy(w.m_big).cuda()
        return _gravity(x, m)
    return None


def _gravity(xv, m):
    """Sum over big bodies of -G m K(s)/s^3 d, K the quintic changeover between
    0.1 and 1 times the larger changeover radius (3 Hill radii)."""
    nb, n = m.numel(), xv.shape[1]
    gm = W.G * (1.0 + m)
    r = xv[:3, :nb].square().sum(0).sqrt()
    a = 1.0 / (2.0 / r - xv[3:, :nb].square().sum(0) / gm)
    rcb = 3.0 * a * (m / 3.0) ** (1.0 / 3.0)
    out = torch.empty((3, n), dtype=torch.float64, device=xv.device)
    chunk = max(1, (1 << 24) // max(1, nb))
    for lo in range(0, n, chunk):
        hi = min(n, lo + chunk)
        d = xv[:3, lo:hi, None] - xv[:3, None, :nb]
        s2 = d.square().sum(0)
        s = s2.sqrt()
        rc = rcb[None, :].expand(hi - lo, nb).clone()
        if lo < nb:
            own = rcb[lo:min(hi, nb)]
            rc[:own.numel()] = torch.maximum(rc[:own.numel()], own[:, None])
        q = ((s - 0.1 * rc) / (0.9 * rc)).clamp(0.0, 1.0)
        f = W.G * m[None, :] * (q * q * q * (q * (6.0 * q - 15.0) + 10.0)) / (s2 * s)
        f = torch.where(s2 > 0, f, torch.zeros_like(f))
        out[:, lo:hi] = -(f[None] * d).sum(2)
    return out


def _kepler(xv, mu, h):
    """Elliptic Kepler motion by h from the difference of eccentric anomalies
    (Gauss f and g)."""
    x, v = xv[:3], xv[3:]
    r = x.square().sum(0).sqrt()
    a = 1.0 / (2.0 / r - v.square().sum(0) / mu)
    n = torch.sqrt(mu / a) / a
    es, ec = (x * v).sum(0) / torch.sqrt(mu * a), 1.0 - r / a
    D = n * h
    for _ in range(50):   # D - ec sin D + es (1 - cos D) = n h
        s, c1 = torch.sin(D), 2.0 * torch.sin(0.5 * D).square()
        D = D - (D - ec * s + es * c1 - n * h) / (1.0 - ec * (1.0 - c1) + es * s)
    s, c1 = torch.sin(D), 2.0 * torch.sin(0.5 * D).square()
    rn = a * (1.0 - ec * (1.0 - c1) + es * s)
    f, g = 1.0 - (a / r) * c1, h + (s - D) / n
    fd, gd = -torch.sqrt(mu * a) * s / (rn * r), 1.0 - (a / rn) * c1
    return torch.cat([f * x + g * v, fd * x + gd * v])
