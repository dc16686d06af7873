"""The work that users of this framework have it do, as cases that can be timed.

Every case is a stretch of a time loop (or one whole differentiable call) through the public Python API.
The material, the 100 m grid (50 m for the TPV3 plane), the time step dt = 0.3 dx / c_p, the boundary grids,
slab thicknesses, history cutoffs and fault parameters are those of this repository's benchmark and tests.

Boundary displacement histories are sums of R separable terms U_r(x) g_r(t) with a k^-2 spatial falloff and
band-limited signals that start from rest, as in the benchmark.  ``prepare`` fills a handle's whole history
with them under a very short truncation window (which stores every step's spectra and skips the long sums),
then restores the uniform cutoff: what a program has in hand in the middle of a long run.

``exact`` evaluates the same sequence in 64 bits with plain torch: FFTs, kernels from Gauss-Legendre
quadrature of their real-axis densities, trapezoid convolution, element-by-element FEM.
"""
import math

import torch

from paper_2102_08756_gb300 import sbim as B
from paper_2102_08756_gb300.autograd import hybrid_rupture, sbim_sequence
from paper_2102_08756_gb300.fault import FaultSolver
from paper_2102_08756_gb300.hybrid import Hybrid
from paper_2102_08756_gb300.sbim import SBIM

CS, CP, RHO = 3464.0, 6000.0, 2670.0
ETA, MU = CP / CS, RHO * CS * CS
MU_K, SIGMA0, MU_S, TAU0 = 0.525, 120e6, 0.677, 70e6
TERMS = 4
DEV = "cuda"


# ---------------------------------------------------------------------------- the cases
def listed():
    return [
        # the plain FP64 method at the size of the small comparison run: launch latency
        dict(name="step_64_fp64", kind="step", n1=64, n3=64, dx=100.0, n_cut=256, precision="fp64",
             kahan=False, steps=16),
        # one half-space of the gradient configuration, stepped by a host program
        dict(name="step_256_fp32", kind="step", n1=256, n3=256, dx=100.0, n_cut=1024,
             precision="fp32", kahan=True, steps=16),
        # the bandwidth configuration: 52 GB of history
        dict(name="step_1024_fp32", kind="step", n1=1024, n3=1024, dx=100.0, n_cut=4096,
             precision="fp32", kahan=True, steps=8),
        # a plane whose sides are no powers of two, hi-only BF16 history
        dict(name="step_360x250_bf16", kind="step", n1=360, n3=250, dx=100.0, n_cut=777,
             precision="bf16", kahan=False, steps=9),
        # the reverse sweep over boundary displacements, BF16 hi/lo history
        dict(name="adjoint_512_bf16x2", kind="adjoint", n1=512, n3=512, dx=100.0, n_cut=1500,
             precision="bf16x2", kahan=True, steps=8),
        # a finite-element program on the host that hands its boundary over every step (pinned buffers)
        dict(name="host_512_fp32", kind="host", n1=512, n3=512, dx=100.0, n_cut=1024,
             precision="fp32", kahan=True, steps=4),
        # the coupled configuration: FEM slab with a fault between two half-spaces
        dict(name="hybrid_512x16x512", kind="hybrid", n1=512, n2=16, n3=512, dx=100.0, n_cut=2000,
             precision="fp32", steps=8),
        # a ragged ensemble of coupled scenarios replayed from a captured graph
        dict(name="ensemble_6", kind="ensemble", members=6, draw_seed=4000, dx=100.0, steps=4),
        # the boundary-only TPV3 solver (symmetry plane) on its rectangular plane
        dict(name="fault_1024x512", kind="fault", n1=1024, n3=512, dx=50.0, n_cut=1600,
             precision="fp32", symmetric=True, steps=6),
        # gradient of a traction misfit with respect to a short boundary history: a whole call
        dict(name="sequence_128", kind="sequence", n1=128, n3=128, dx=100.0, n_cut=48,
             precision="fp32", steps=64),
        # gradient of a coupled rupture with respect to Dc, checkpointed: a whole call
        dict(name="rupture_64x8x64", kind="rupture", n1=64, n2=8, n3=64, dx=100.0, n_cut=40,
             steps=48, every=12),
        # the allocation-free entry point on a caller's own spectra
        dict(name="noalloc_256", kind="noalloc", n1=256, n3=256, dx=100.0, n_lags=500),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _even(rng, lo, hi):
    return max(2, 2 * (_log(rng, lo, hi) // 2))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "adjoint", "host", "hybrid", "ensemble", "fault",
                       "sequence", "rupture", "noalloc"])
    n1 = _even(rng, 16, 1024)
    n3 = n1 if rng.random() < 0.5 else _even(rng, max(16, n1 // 4), min(1024, 4 * n1))
    n_cut = _log(rng, 16, 4096)
    if kind in ("step", "adjoint", "host"):
        precision = rng.choice(["fp32", "fp32", "bf16x2", "bf16", "fp64"])
        if precision == "fp64":
            n1, n3, n_cut = min(n1, 256), min(n3, 256), min(n_cut, 512)
        return dict(kind=kind, n1=n1, n3=n3, dx=100.0, n_cut=n_cut, precision=precision,
                    kahan=precision != "bf16" and precision != "fp64", steps=rng.randint(1, 8))
    if kind == "hybrid":
        return dict(kind=kind, n1=min(n1, 512), n2=2 * rng.randint(2, 8), n3=min(n3, 512), dx=100.0,
                    n_cut=min(n_cut, 2000), precision=rng.choice(["fp32", "fp32", "fp32", "fp64"])
                    if n1 * n3 <= 128 * 128 and n_cut <= 512 else "fp32", steps=rng.randint(1, 6))
    if kind == "ensemble":
        return dict(kind=kind, members=rng.randint(2, 6), draw_seed=rng.randint(0, 10 ** 6), dx=100.0,
                    steps=rng.randint(1, 4))
    if kind == "fault":
        return dict(kind=kind, n1=n1, n3=min(n3, 512), dx=50.0, n_cut=min(n_cut, 1600),
                    precision="fp32", symmetric=rng.random() < 0.5, steps=rng.randint(1, 6))
    if kind == "sequence":
        return dict(kind=kind, n1=min(n1, 256), n3=min(n3, 256), dx=100.0, n_cut=rng.randint(16, 64),
                    precision="fp32", steps=rng.randint(8, 64))
    if kind == "rupture":
        return dict(kind=kind, n1=2 * rng.randint(16, 48), n2=2 * rng.randint(2, 6),
                    n3=2 * rng.randint(16, 48), dx=100.0, n_cut=rng.randint(12, 48),
                    steps=rng.randint(12, 48), every=rng.randint(4, 16))
    return dict(kind="noalloc", n1=min(n1, 512), n3=min(n3, 512), dx=100.0, n_lags=min(n_cut, 600))


# ---------------------------------------------------------------------------- inputs
def _gen(seed, k=0):
    return torch.Generator(device=DEV).manual_seed(1000003 * int(seed) + k)


def _dt(dx):
    return 0.3 * dx / CP


class _Separable:
    """u(x, t_n) = sum_r g[r, n] U_r(x) in 64 bits; U [R, 3, n3, n1]."""

    def __init__(self, n1, n3, dx, steps, seed, rms=1e-3):
        g = _gen(seed)
        j1 = torch.arange(n1 // 2 + 1, device=DEV, dtype=torch.float64)[None, :] / n1
        j3 = torch.fft.fftfreq(n3, device=DEV, dtype=torch.float64)[:, None]
        fall = 1.0 / (1.0 + (j1 ** 2 + j3 ** 2) * 32.0 ** 2)       # k^-2 beyond 32 grid spacings
        z = torch.randn((TERMS, 3, n3, n1 // 2 + 1, 2), generator=g, device=DEV, dtype=torch.float64)
        U = torch.fft.irfft2(torch.view_as_complex(z) * fall, s=(n3, n1))
        self.U = U * (rms / (U.square().mean().sqrt() * math.sqrt(TERMS)))
        t = torch.arange(steps, device=DEV, dtype=torch.float64)
        w = (0.05 + 0.95 * torch.rand((TERMS, 8), generator=g, device=DEV, dtype=torch.float64))
        w *= 0.25 * math.pi / dx * CS * _dt(dx)                    # up to a quarter of Nyquist
        ph = 2 * math.pi * torch.rand((TERMS, 8), generator=g, device=DEV, dtype=torch.float64)
        amp = torch.randn((TERMS, 8), generator=g, device=DEV, dtype=torch.float64)
        sig = (amp[:, :, None] * torch.sin(w[:, :, None] * t + ph[:, :, None])).sum(1)
        self.g = sig * torch.sin(0.5 * math.pi * torch.clamp(t / 20.0, max=1.0)) ** 2
        self.dt = _dt(dx)

    def u(self, n):
        return torch.tensordot(self.g[:, n], self.U, dims=1)

    def v(self, n):
        prev = self.g[:, n - 1] if n > 0 else torch.zeros_like(self.g[:, 0])
        return torch.tensordot((self.g[:, n] - prev) / self.dt, self.U, dims=1)


def _fill_steps(n_cut):
    return n_cut + 5          # past the cutoff: the ring has wrapped


def _real(precision):
    return torch.float64 if precision == "fp64" else torch.float32


def _fill(handle, sep, n_fill, dtype, adjoint=False, sign=1.0):
    """Give a handle the history sign * u(0..n_fill-1)."""
    n3, n1 = sep.U.shape[-2:]
    B.sbim_set_window(handle, 1e-6)
    zero = torch.zeros((3, n3, n1), dtype=dtype, device=DEV)
    out, out2 = torch.empty_like(zero), torch.empty_like(zero)
    flat = (sign * sep.U).reshape(TERMS, -1)
    for n0 in range(0, n_fill, 64):
        k = min(64, n_fill - n0)
        us = (sep.g[:, n0:n0 + k].T @ flat).to(dtype).reshape(k, 3, n3, n1)
        for i in range(k):
            if adjoint:
                B.sbim_step_adjoint(handle, us[i].data_ptr(), out.data_ptr(), out2.data_ptr())
            else:
                B.sbim_step(handle, us[i].data_ptr(), zero.data_ptr(), out.data_ptr())
        torch.cuda.current_stream().synchronize()
    B.sbim_set_window(handle, 0.0)


def _law(n1, n3, dx, seed, dc=0.4):
    """TPV3-like friction: a square overstressed patch in a uniform prestress (64 bits, CPU)."""
    r = torch.Generator().manual_seed(int(seed))
    c1 = (torch.arange(n1, dtype=torch.float64) - n1 / 2 + 0.5)[None, :]
    c3 = (torch.arange(n3, dtype=torch.float64) - n3 / 2 + 0.5)[:, None]
    half = max(2.0, min(15.0, min(n1, n3) / 6.0))
    patch = (c1.abs() <= half) & (c3.abs() <= half)
    base = TAU0 * (0.97 + 0.06 * torch.rand((), generator=r, dtype=torch.float64))
    tau0 = torch.where(patch, torch.tensor(1.005 * MU_S * SIGMA0, dtype=torch.float64), base)
    return dict(mu_s=torch.full((n3, n1), MU_S, dtype=torch.float64), tau0=tau0, mu_k=MU_K, Dc=dc,
                sigma0=SIGMA0)


def _scenarios(case):
    """The ensemble's members: grids from {128, 256, 384, 512}^2, slabs of 8-16 elements, cutoffs
    512-2000, Dc 0.2-0.8 m, seeded as the case says."""
    r = torch.Generator().manual_seed(int(case["draw_seed"]))
    ri = lambda lo, hi: int(torch.randint(lo, hi + 1, (), generator=r))  # noqa: E731
    return [dict(n1=n, n3=n, n2=2 * ri(4, 8), n_cut=ri(512, 2000), dx=case["dx"],
                 Dc=0.2 + 0.6 * float(torch.rand((), generator=r, dtype=torch.float64)))
            for n in ((128, 256, 384, 512)[ri(0, 3)] for _ in range(case["members"]))]


def _slab_state(c, sep, n, dtype):
    """u, v, a of a slab whose boundaries carry the half-spaces' displacements at step n: the two
    sides of the fault move in opposite senses, with an amplitude that varies across the slab."""
    L, f = c["n2"] + 2, c["n2"] // 2
    w = torch.tensor([1.0 - 0.02 * (L - 1 - l) if l > f else -(1.0 - 0.02 * l) for l in range(L)],
                     device=DEV, dtype=torch.float64)[:, None, None, None]
    a = (sep.v(n) - sep.v(n - 1)) / sep.dt
    return [(w * x).to(dtype).contiguous() for x in (sep.u(n), sep.v(n), a)]


class _Closing:
    """Closes what a state holds, in order, when the state goes."""

    def __init__(self, *calls):
        self.calls = calls

    def __del__(self):
        for f in self.calls:
            try:
                f()
            except Exception:
                pass


def _hybrid(c, seed, stream, precision):
    dt, dtype = _dt(c["dx"]), _real(precision)
    h = Hybrid(c["n1"], c["n2"], c["n3"], c["dx"], CS, CP, RHO, dt, c["n_cut"], precision, True, True,
               stream=stream)
    law = _law(c["n1"], c["n3"], c["dx"], seed, c.get("Dc", 0.4))
    h.set_fault(law["mu_s"].numpy(), law["tau0"].numpy(), law["mu_k"], law["Dc"], law["sigma0"])
    n = _fill_steps(c["n_cut"])
    sep = _Separable(c["n1"], c["n3"], c["dx"], n, seed, rms=0.05)
    _, _, top, bot = B.sbim_hybrid_info(h.h)
    _fill(top, sep, n, dtype)
    _fill(bot, sep, n, dtype, sign=-1.0)
    h.set_state(*_slab_state(c, sep, n - 1, dtype))
    stream.synchronize()
    return h


def prepare(case, seed):
    kind = case["kind"]
    S = case.get("steps", 1)
    st = {"case": case}
    if kind in ("step", "adjoint", "host"):
        n1, n3, dx, n_cut = case["n1"], case["n3"], case["dx"], case["n_cut"]
        dtype = _real(case["precision"])
        n = _fill_steps(n_cut)
        sep = _Separable(n1, n3, dx, n + S, seed)
        st["h"] = SBIM(n1, n3, n1 * dx, n3 * dx, CS, CP, RHO, _dt(dx), n_cut, 1, case["precision"],
                       case["kahan"])
        _fill(st["h"].h, sep, n, dtype, adjoint=kind == "adjoint")
        u = torch.stack([sep.u(n + s) for s in range(S)]).to(dtype)
        v = torch.stack([sep.v(n + s) for s in range(S)]).to(dtype)
        if kind == "host":
            u, v = u.cpu().pin_memory(), v.cpu().pin_memory()
            out = torch.empty_like(u).pin_memory()
            st.update(keep=(u, v, out), u=u.numpy(), v=v.numpy(), out=out.numpy())
        else:
            st.update(u=u, v=v, out=torch.empty_like(u), out2=torch.empty_like(u))
    elif kind == "hybrid":
        stream = torch.cuda.current_stream()
        st["h"] = _hybrid(case, seed, stream, case["precision"])
    elif kind == "ensemble":
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            hs = [_hybrid(c, seed + 17 * i, stream, "fp32") for i, c in enumerate(_scenarios(case))]
            b = B.sbim_hybrid_batch_create([x.h for x in hs])
            B.sbim_hybrid_batch_capture(b)
            stream.synchronize()
        st.update(b=b, hs=hs, stream=stream,
                  closing=_Closing(lambda: B.sbim_hybrid_batch_destroy(b), *[x.close for x in hs]))
    elif kind == "fault":
        n1, n3, dx, n_cut = case["n1"], case["n3"], case["dx"], case["n_cut"]
        n = _fill_steps(n_cut)
        sep = _Separable(n1, n3, dx, n, seed, rms=0.05)
        h = FaultSolver(n1, n3, n1 * dx, n3 * dx, CS, CP, RHO, _dt(dx), n_cut, case["precision"],
                        symmetric=case["symmetric"])
        law = _law(n1, n3, dx, seed)
        h.set_fault(law["mu_s"].numpy(), law["tau0"].numpy(), law["mu_k"], law["Dc"], law["sigma0"])
        up, lo = h.handles()
        dtype = _real(case["precision"])
        _fill(up, sep, n, dtype)
        if lo is not None:
            _fill(lo, sep, n, dtype, sign=-1.0)
        u, v = sep.u(n - 1), sep.v(n - 1)
        h.set_state(torch.stack([u, -u]).to(dtype), torch.stack([v, -v]).to(dtype))
        st["h"] = h
    elif kind == "sequence":
        n1, n3, dx = case["n1"], case["n3"], case["dx"]
        dtype = _real(case["precision"])
        sep = _Separable(n1, n3, dx, S, seed)
        st["u"] = torch.stack([sep.u(s) for s in range(S)]).to(dtype).requires_grad_()
        st["v"] = torch.stack([sep.v(s) for s in range(S)]).to(dtype).requires_grad_()
        st["bar"] = torch.randn(st["u"].shape, generator=_gen(seed, 5), device=DEV, dtype=dtype)
        st["p"] = dict(n1=n1, n3=n3, L1=n1 * dx, L3=n3 * dx, cs=CS, cp=CP, rho=RHO, dt=_dt(dx),
                       n_cut=case["n_cut"], side=1, precision=case["precision"])
    elif kind == "rupture":
        law = _law(case["n1"], case["n3"], case["dx"], seed)
        st["dc"] = torch.tensor(0.05, dtype=torch.float32, device=DEV, requires_grad=True)
        st["bar"] = torch.randn((S, 3, case["n3"], case["n1"]), generator=_gen(seed, 5), device=DEV)
        st["p"] = dict(n1=case["n1"], n2=case["n2"], n3=case["n3"], h=case["dx"], cs=CS, cp=CP, rho=RHO,
                       dt=_dt(case["dx"]), n_cut=case["n_cut"], mu_s=law["mu_s"].numpy(),
                       tau0=law["tau0"].numpy(), mu_k=MU_K, sigma0=SIGMA0, steps=S,
                       every=case["every"])
    else:
        st["x"] = _noalloc_input(case, seed)
        st["out"] = torch.empty((3, case["n3"], case["n1"] // 2 + 1), dtype=torch.complex64, device=DEV)
    return st


def _noalloc_input(case, seed):
    """Displacement spectra of the last n_lags steps, newest first: [n_lags, 3, n3, n1/2+1]."""
    sep = _Separable(case["n1"], case["n3"], case["dx"], case["n_lags"] + 30, seed)
    flat = torch.fft.rfft2(sep.U).reshape(TERMS, -1)
    g = sep.g[:, 30:].flip(1).T.to(flat.dtype)
    return (g @ flat).to(torch.complex64).reshape(-1, 3, case["n3"], case["n1"] // 2 + 1).contiguous()


# ---------------------------------------------------------------------------- one pass
def run(state):
    case = state["case"]
    kind, S = case["kind"], case.get("steps", 1)
    if kind == "step":
        for s in range(S):
            state["h"].step(state["u"][s], state["v"][s], state["out"][s])
        return state["out"]
    if kind == "adjoint":
        for s in range(S):
            state["h"].step_adjoint(state["u"][s], state["out"][s], state["out2"][s])
        return state["out"], state["out2"]
    if kind == "host":
        for s in range(S):
            state["h"].step_host(state["u"][s], state["v"][s], state["out"][s])
        return state["out"]
    if kind == "hybrid":
        for _ in range(S):
            state["h"].step()
        return state["h"].get_state(), state["h"].fault_fields(), state["h"].boundary_tractions()
    if kind == "ensemble":
        with torch.cuda.stream(state["stream"]):
            for _ in range(S):
                B.sbim_hybrid_batch_replay(state["b"])
            out = [(x.get_state(), x.fault_fields()) for x in state["hs"]]
        torch.cuda.current_stream().wait_stream(state["stream"])
        return out
    if kind == "fault":
        for _ in range(S):
            state["h"].step()
        return state["h"].get_state(), state["h"].fault_fields()
    if kind == "sequence":
        u, v = state["u"], state["v"]
        u.grad = v.grad = None
        tau = sbim_sequence(u, v, **state["p"])
        tau.backward(state["bar"])
        return tau.detach(), u.grad, v.grad
    if kind == "rupture":
        dc = state["dc"]
        dc.grad = None
        tau = hybrid_rupture(dc, **state["p"])
        tau.backward(state["bar"])
        return tau.detach(), dc.grad
    n1, n3, dx = case["n1"], case["n3"], case["dx"]
    B.sbim_spectral_response_noalloc(n1, n3, n1 * dx, n3 * dx, CS, CP, RHO, _dt(dx), 1, case["n_lags"],
                                     state["x"].data_ptr(), state["out"].data_ptr(),
                                     torch.cuda.current_stream().cuda_stream)
    return state["out"]


# ---------------------------------------------------------------------------- what a pass cannot do without
def _half_space(n1, n3, lags, steps, rec, real):
    """Bytes and flops of `steps` consecutive updates that reach `lags` steps back: the stored
    history read once, the new spectra stored, u, v and tau of every step; 5 real x complex
    multiply-adds per mode and lag and the transforms of 6 planes."""
    bins, plane = n3 * (n1 // 2 + 1), n1 * n3
    b = bins * 3 * rec * (max(0, lags - 1) + steps) + 9 * plane * real * steps
    f = steps * (20.0 * bins * lags + 6 * 2.5 * plane * math.log2(plane))
    return b, f


_REC = {"fp64": 16, "fp32": 8, "bf16x2": 8, "bf16": 4}


def _slab(c, steps, real):
    nodes = c["n1"] * c["n3"] * (c["n2"] + 2)
    return 2 * 9 * nodes * real, steps * nodes * (2.0 * 236 + 40)


def work(case):
    kind, S = case["kind"], case.get("steps", 1)
    if kind in ("step", "adjoint", "host"):
        b, f = _half_space(case["n1"], case["n3"], case["n_cut"], S, _REC[case["precision"]],
                           8 if case["precision"] == "fp64" else 4)
    elif kind in ("hybrid", "ensemble"):
        b = f = 0.0
        for c in ([case] if kind == "hybrid" else _scenarios(case)):
            p = c.get("precision", "fp32")
            r = 8 if p == "fp64" else 4
            hb, hf = _half_space(c["n1"], c["n3"], c["n_cut"], S, _REC[p], r)
            sb, sf = _slab(c, S, r)
            b, f = b + 2 * hb + sb, f + 2 * hf + sf
    elif kind == "fault":
        hb, hf = _half_space(case["n1"], case["n3"], case["n_cut"], S, _REC[case["precision"]], 4)
        k = 1 if case["symmetric"] else 2
        b, f = k * hb + 24 * case["n1"] * case["n3"] * 4, k * hf
    elif kind == "sequence":
        hb, hf = _half_space(case["n1"], case["n3"], 1, S, 8, 4)
        pairs = sum(min(n + 1, case["n_cut"]) for n in range(S))
        bins = case["n3"] * (case["n1"] // 2 + 1)
        b, f = 2 * hb, 2 * (hf + 20.0 * bins * (pairs - S))
    elif kind == "rupture":
        hb, hf = _half_space(case["n1"], case["n3"], 1, S, 8, 4)
        pairs = sum(min(n + 1, case["n_cut"]) for n in range(S))
        bins = case["n3"] * (case["n1"] // 2 + 1)
        sb, sf = _slab(case, 3 * S, 4)
        b = 4 * hb + sb + S * 3 * case["n1"] * case["n3"] * 8
        f = 4 * (hf + 20.0 * bins * (pairs - S)) + sf
    else:
        bins = case["n3"] * (case["n1"] // 2 + 1)
        b, f = bins * 24.0 * (case["n_lags"] + 1), 32.0 * bins * case["n_lags"]
    return {"bytes": float(b), "flops": float(f)}


# ---------------------------------------------------------------------------- 64-bit values
def _gauss(n_panels, width):
    """16-point Gauss-Legendre nodes and weights on [0, width], n_panels panels."""
    k = torch.arange(1, 16, dtype=torch.float64)
    off = k / torch.sqrt(4 * k * k - 1)
    ev, vec = torch.linalg.eigh(torch.diag(off, 1) + torch.diag(off, -1))
    x, w = ev.to(DEV), (2 * vec[0] ** 2).to(DEV)
    hw = 0.5 * width / n_panels
    mid = hw * (2 * torch.arange(n_panels, device=DEV, dtype=torch.float64) + 1)
    return (mid[:, None] + hw * x).reshape(-1), (hw * w).repeat(n_panels)


def _kernels(T):
    """H11, H22, H33, H12 at the points T >= 0: cosine / sine transforms of their densities."""
    out = torch.empty((T.numel(), 4), device=DEV, dtype=torch.float64)
    order = torch.argsort(T)
    i = 0
    while i < T.numel():
        k = min(T.numel(), i + 4096)
        idx = order[i:k]
        t = T[idx][:, None]
        pan = int(float(t.max()) * ETA * 0.5 * math.pi / 5.0) + 4
        th, w = _gauss(pan, 0.5 * math.pi)
        y, b = torch.sin(th), torch.cos(th)                        # 0 <= y <= 1
        a = torch.sqrt(1 - y * y / ETA ** 2)
        gg = (1 + a * b) / (1 + (1 - y * y) / ETA ** 2)
        low = torch.stack([a * gg, b * gg, b], 1) * (w * b)[:, None]
        s, c = torch.sin(th), torch.cos(th)                        # 1 <= y <= eta
        yu = 1 + (ETA - 1) * s * s
        Bq = math.sqrt(ETA - 1) * s * torch.sqrt(yu + 1)
        A = math.sqrt(ETA - 1) * c * torch.sqrt(ETA + yu) / ETA
        f = A * yu * yu / (1 + A * A * Bq * Bq) * (2 * (ETA - 1) * s * c) * w
        up = torch.stack([f, -f * Bq * Bq], 1)
        cl, cu, su = torch.cos(t * y), torch.cos(t * yu), torch.sin(t * yu)
        r = torch.cat([cl @ low, (su @ (f * Bq))[:, None]], 1)
        r[:, :2] += cu @ up
        out[idx] = r * (2 / math.pi)
        i = k
    return out


class _Kernel:
    """The kernels on a grid T_j = j h, 10-point Lagrange interpolation in between (the kernels are
    entire, H11, H22, H33 even and H12 odd)."""

    H, N = 1.0 / 24.0, 10

    def __init__(self, t_max):
        j = torch.arange(-5, int(t_max / self.H) + 8, device=DEV, dtype=torch.float64)
        self.v = _kernels(j.abs() * self.H)
        self.v[:, 3] *= torch.sign(j)
        off = torch.arange(-4, 6, device=DEV, dtype=torch.float64)
        self.off = off
        self.den = torch.stack([torch.prod(torch.cat([off[:k], off[k + 1:]]).neg() + off[k])
                                for k in range(self.N)])

    def __call__(self, T):
        """[4, *T.shape]"""
        x = T.reshape(-1) / self.H
        i = torch.floor(x)
        d = (x - i)[:, None] - self.off
        out = torch.zeros((x.numel(), 4), device=DEV, dtype=torch.float64)
        i = i.long() + 5
        for k in range(self.N):
            o = torch.cat([d[:, :k], d[:, k + 1:]], 1).prod(1) / self.den[k]
            out += o[:, None] * self.v[i + (k - 4)]
        return out.T.reshape(4, *T.shape)


class _HalfSpace:
    """The traction update in 64 bits: an old separable history (or none) and new spectra."""

    def __init__(self, n1, n3, dx, n_cut, side, sep=None, n_old=0, n_new=1, sign=1.0, kern=None):
        self.n1, self.n3, self.side, self.n_cut = n1, n3, side, n_cut
        j1 = torch.arange(n1 // 2 + 1, device=DEV, dtype=torch.float64)[None, :].expand(n3, -1)
        r3 = torch.arange(n3, device=DEV, dtype=torch.float64)[:, None].expand(-1, n1 // 2 + 1)
        j3 = torch.where(r3 <= n3 // 2, r3, r3 - n3)
        k1, k3 = 2 * math.pi / (n1 * dx) * j1.reshape(-1), 2 * math.pi / (n3 * dx) * j3.reshape(-1)
        self.q = torch.sqrt(k1 * k1 + k3 * k3)
        qs = torch.where(self.q > 0, self.q, torch.ones_like(self.q))
        e1, e3 = k1 / qs, k3 / qs
        ny1, ny3 = j1.reshape(-1) == n1 // 2, j3.reshape(-1) == n3 // 2
        zero = torch.zeros_like(e1)
        self.e11, self.e33 = e1 * e1, e3 * e3
        self.e13 = torch.where(ny1 | ny3, zero, e1 * e3)
        self.c1, self.c3 = torch.where(ny1, zero, e1), torch.where(ny3, zero, e3)
        uq, self.cls = torch.unique(self.q, return_inverse=True)
        self.dT = uq * (CS * _dt(dx))
        kern = kern or _Kernel(float(self.dT.max()) * max(n_cut - 1, n_new) + 1)
        self.w_new = self.weights(kern, torch.arange(min(n_new, n_cut), device=DEV))
        self.z_old = None
        if sep is not None:
            # [4, class, r, s]: sum over the lags that reach the old steps 0 .. n_old-1
            S = n_new
            self.z_old = torch.empty((4, uq.numel(), TERMS * S), device=DEV, dtype=torch.float64)
            m = torch.arange(1, n_cut, device=DEV)
            t = n_old + torch.arange(S, device=DEV)[None, :] - m[:, None]        # [m, s]
            ok = (t < n_old) & (t >= 0)
            G = torch.where(ok[None], sep.g[:, t.clamp(0, n_old - 1)], 0.0)       # [r, m, s]
            G = G.permute(1, 0, 2).reshape(n_cut - 1, TERMS * S)
            step = max(1, 3_000_000 // max(1, n_cut))
            for i in range(0, uq.numel(), step):
                T = self.dT[i:i + step, None] * m
                self.z_old[:, i:i + step] = (kern(T) * self.dT[i:i + step, None]) @ G
            self.Uh = sign * torch.fft.rfft2(sep.U).reshape(TERMS, 3, -1)
        self.new = []

    def weights(self, kern, m):
        w = kern(self.dT[:, None] * m) * self.dT[:, None]
        w[..., 0] *= torch.where(m[:1] == 0, 0.5, 1.0)
        return w

    def _put(self, D):
        self.new = self.new + [D]

    def rewind(self):
        self.new = self.new[:-1]

    def s(self, u):
        """The non-local traction s at the next step, for the displacement u there."""
        D = torch.fft.rfft2(u).reshape(3, -1)
        self._put(D)
        s = len(self.new) - 1
        Z = 0
        for lag in range(min(s + 1, self.n_cut)):
            Z = Z + self.w_new[:, self.cls, lag][:, None] * self.new[s - lag]
        if self.z_old is not None:
            zo = self.z_old.reshape(4, -1, TERMS, self.z_old.shape[2] // TERMS)[..., s][:, self.cls]
            Z = Z + torch.einsum("aqr,rcq->acq", zo.to(D.dtype), self.Uh)
        return torch.fft.irfft2(self.operator(Z, D).reshape(3, self.n3, -1), s=(self.n3, self.n1))

    def operator(self, Z, D):
        mq, sd, inst = MU * self.q, self.side, 2 - ETA
        p = [inst * D[c] + Z[3, c] for c in range(3)]
        f1 = -sd * mq * (self.e11 * Z[0, 0] + self.e13 * (Z[0, 2] - Z[2, 2]) + self.e33 * Z[2, 0])
        f3 = -sd * mq * (self.e13 * (Z[0, 0] - Z[2, 0]) + self.e33 * Z[0, 2] + self.e11 * Z[2, 2])
        f1 = f1 + 1j * mq * self.c1 * p[1]
        f3 = f3 + 1j * mq * self.c3 * p[1]
        f2 = -1j * mq * (self.c1 * p[0] + self.c3 * p[2]) - sd * mq * Z[1, 1]
        return torch.stack([f1, f2, f3])

    def damping(self, v):
        return -self.side * MU / CS * _imp() * v

    def tau(self, u, v):
        return self.damping(v) + self.s(u)


def _imp():
    return torch.tensor([1.0, ETA, 1.0], device=DEV, dtype=torch.float64)[:, None, None]


def _mag(x, y):
    z = x * x + y * y
    pos = z > 0
    return torch.where(pos, torch.sqrt(torch.where(pos, z, torch.ones_like(z))), torch.zeros_like(z))


def _slipweak(law, dc, stick, slip):
    """The fault traction of the stick / slip law."""
    mu_s, tau0 = law["mu_s"].to(DEV), law["tau0"].to(DEV)
    mu_k = law["mu_k"]
    fric = torch.where(slip < dc, mu_s - (mu_s - mu_k) * slip / dc, torch.full_like(mu_s, mu_k))
    strength = (law["sigma0"] - stick[1]) * fric
    t1, t3 = tau0 + stick[0], stick[2]
    mag = _mag(t1, t3)
    k = torch.where(mag > strength, strength / mag, torch.ones_like(mag))
    return torch.stack([t1 * k - tau0, stick[1], t3 * k])


def _rounded(law):
    """The maps as an FP32 handle holds them."""
    return dict(law, mu_s=law["mu_s"].float().double(), tau0=law["tau0"].float().double())


class _Slab:
    """The coupled step in 64 bits (element-by-element forces)."""

    def __init__(self, c, law, dc, top, bot, state=None):
        self.c, self.law, self.dc, self.top, self.bot = c, law, dc, top, bot
        n1, n2, n3, h = c["n1"], c["n2"], c["n3"], c["dx"]
        self.h, self.f, self.L, self.dt = h, n2 // 2, n2 + 2, _dt(h)
        self.K = _hex8(h).to(DEV)
        self.elem = [l for l in range(self.L - 1) if l != self.f]      # lower layer of each element layer
        m = torch.zeros(self.L, device=DEV, dtype=torch.float64)
        for l in self.elem:
            m[l] += 0.5 * RHO * h ** 3
            m[l + 1] += 0.5 * RHO * h ** 3
        self.m = m[:, None, None, None]
        shape = (self.L, 3, n3, n1)
        z = torch.zeros(shape, device=DEV, dtype=torch.float64)
        self.u, self.v, self.a = [x.double() for x in state] if state else (z, z, z)

    def force(self, u):
        """-K u"""
        out = []
        add = [0] * self.L
        for l in self.elem:
            x = []
            for a in range(8):
                w = u[l + ((a >> 1) & 1)]
                x.append(torch.roll(w, (-(a >> 2), -(a & 1)), (1, 2)))
            x = torch.stack(x).reshape(24, -1)
            y = (self.K @ x).reshape(8, 3, *u.shape[2:])
            for a in range(8):
                add[l + ((a >> 1) & 1)] = add[l + ((a >> 1) & 1)] - torch.roll(
                    y[a], (a >> 2, a & 1), (1, 2))
        out = torch.stack(add)
        return out

    def step(self):
        dt, A, f = self.dt, self.h ** 2, self.f
        vp = self.v + dt * self.a
        u = self.u + dt * self.v + 0.5 * dt * dt * self.a
        self.tt, self.tb = self.top.tau(u[-1], vp[-1]), self.bot.tau(u[0], vp[0])
        F = self.force(u)
        pad = torch.zeros_like(F[1:-1])
        F = F + torch.cat([-A * self.tb[None], pad, A * self.tt[None]])
        af = F / self.m
        vf = vp - 0.5 * dt * self.a + dt * af
        imp = dt * A * (1 / self.m[f] + 1 / self.m[f + 1])
        stick = (vf[f + 1] - vf[f]) / imp
        d = u[f + 1] - u[f]
        tau = _slipweak(self.law, self.dc, stick, _mag(d[0], d[2]))
        k = A * tau / self.m[f]
        an = torch.cat([af[:f], (af[f] + k)[None], (af[f + 1] - k)[None], af[f + 2:]])
        self.v = vp + 0.5 * dt * (an - self.a)
        self.u, self.a, self.traction = u, an, tau

    def fields(self):
        f = self.f
        return self.u[f + 1] - self.u[f], self.v[f + 1] - self.v[f], self.traction


def _hex8(h):
    lam = RHO * CP ** 2 - 2 * MU
    D = torch.zeros((6, 6), dtype=torch.float64)
    D[:3, :3] = lam
    D[range(3), range(3)] += 2 * MU
    D[range(3, 6), range(3, 6)] = MU
    s = torch.tensor([[1.0 if a >> b & 1 else -1.0 for b in range(3)] for a in range(8)],
                     dtype=torch.float64)
    K = torch.zeros((24, 24), dtype=torch.float64)
    for p in s / math.sqrt(3.0):
        f = 1 + s * p
        dN = torch.stack([s[:, 0] * f[:, 1] * f[:, 2], s[:, 1] * f[:, 0] * f[:, 2],
                          s[:, 2] * f[:, 0] * f[:, 1]], 1) / (4 * h)
        Bm = torch.zeros((6, 24), dtype=torch.float64)
        for i in range(3):
            Bm[i, i::3] = dN[:, i]
        for r, (i, j) in enumerate(((0, 1), (1, 2), (0, 2))):
            Bm[3 + r, i::3] = dN[:, j]
            Bm[3 + r, j::3] = dN[:, i]
        K += Bm.T @ D @ Bm * (h / 2) ** 3
    return K


def _exact_hybrid(c, seed, S, precision):
    n, dtype = _fill_steps(c["n_cut"]), _real(precision)
    sep = _Separable(c["n1"], c["n3"], c["dx"], n, seed, rms=0.05)
    top = _HalfSpace(c["n1"], c["n3"], c["dx"], c["n_cut"], 1, sep, n, S)
    bot = _HalfSpace(c["n1"], c["n3"], c["dx"], 1, -1, None, 0, 1)
    bot.n_cut, bot.z_old, bot.Uh, bot.w_new = top.n_cut, top.z_old, -top.Uh, top.w_new
    law = _law(c["n1"], c["n3"], c["dx"], seed, c.get("Dc", 0.4))
    law = _rounded(law) if precision != "fp64" else law
    x = _Slab(c, law, law["Dc"], top, bot, _slab_state(c, sep, n - 1, dtype))
    for _ in range(S):
        x.step()
    return (x.u, x.v, x.a), x.fields(), (x.tt, x.tb)


def exact(case, seed):
    kind, S = case["kind"], case.get("steps", 1)
    n1, n3, dx = case.get("n1"), case.get("n3"), case["dx"]
    if kind in ("step", "adjoint", "host"):
        n = _fill_steps(case["n_cut"])
        dtype = _real(case["precision"])
        sep = _Separable(n1, n3, dx, n + S, seed)
        hs = _HalfSpace(n1, n3, dx, case["n_cut"], 1, sep, n, S)
        out, out2 = [], []
        for s in range(S):
            u, v = sep.u(n + s).to(dtype).double(), sep.v(n + s).to(dtype).double()
            out.append(hs.s(u) if kind == "adjoint" else hs.tau(u, v))
            if kind == "adjoint":
                out2.append(hs.damping(u))
        return (torch.stack(out), torch.stack(out2)) if kind == "adjoint" else torch.stack(out)
    if kind == "hybrid":
        return _exact_hybrid(case, seed, S, case["precision"])
    if kind == "ensemble":
        return [_exact_hybrid(c, seed + 17 * i, S, "fp32")[:2] for i, c in enumerate(_scenarios(case))]
    if kind == "fault":
        n = _fill_steps(case["n_cut"])
        dtype = _real(case["precision"])
        sep = _Separable(n1, n3, dx, n, seed, rms=0.05)
        up = _HalfSpace(n1, n3, dx, case["n_cut"], 1, sep, n, S)
        lo = None
        if not case["symmetric"]:
            lo = _HalfSpace(n1, n3, dx, 1, -1, None, 0, 1)
            lo.n_cut, lo.z_old, lo.Uh, lo.w_new = up.n_cut, up.z_old, -up.Uh, up.w_new
        law, dt, z = _rounded(_law(n1, n3, dx, seed)), _dt(dx), MU / CS * _imp()
        flip = torch.tensor([-1.0, 1.0, -1.0], device=DEV, dtype=torch.float64)[:, None, None]
        u0, v0 = sep.u(n - 1), sep.v(n - 1)
        u, v = (torch.stack([x, -x]).to(dtype).double() for x in (u0, v0))
        if lo is None:
            u[1], v[1] = flip * u[0], flip * v[0]

        def solve(x):
            a = up.s(x[0])
            b = lo.s(x[1]) if lo is not None else torch.stack([a[0], -a[1], a[2]])
            stick, vbar = 0.5 * (a + b), (a - b) / (2 * z)
            d = x[0] - x[1]
            tau = _slipweak(law, law["Dc"], stick, _mag(d[0], d[2]))
            V = 2 * (stick - tau) / z[0]
            return torch.stack([vbar + 0.5 * V, vbar - 0.5 * V]), tau, V

        def tied(x):
            return torch.stack([x[0], flip * x[0]]) if lo is None else x

        for _ in range(S):
            vs, _, _ = solve(tied(u + dt * v))
            up.rewind()
            if lo is not None:
                lo.rewind()
            u = tied(u + 0.5 * dt * (v + vs))
            v, tau, V = solve(u)
        return (u, v), (u[0] - u[1], V, tau)
    if kind == "sequence":
        dtype = _real(case["precision"])
        sep = _Separable(n1, n3, dx, S, seed)
        fwd = _HalfSpace(n1, n3, dx, case["n_cut"], 1, None, 0, S)
        rev = _HalfSpace(n1, n3, dx, 1, 1, None, 0, 1)
        rev.n_cut, rev.w_new = fwd.n_cut, fwd.w_new
        bar = torch.randn((S, 3, n3, n1), generator=_gen(seed, 5), device=DEV, dtype=dtype).double()
        tau = torch.stack([fwd.tau(sep.u(s).to(dtype).double(), sep.v(s).to(dtype).double())
                           for s in range(S)])
        ub = [None] * S
        for s in reversed(range(S)):
            ub[s] = rev.s(bar[s])
        return tau, torch.stack(ub), fwd.damping(bar)
    if kind == "rupture":
        law = _rounded(_law(n1, n3, dx, seed))
        dc = torch.tensor(0.05, dtype=torch.float32).double().to(DEV).requires_grad_()
        bar = torch.randn((S, 3, n3, n1), generator=_gen(seed, 5), device=DEV).double()
        top = _HalfSpace(n1, n3, dx, case["n_cut"], 1, None, 0, S)
        bot = _HalfSpace(n1, n3, dx, 1, -1, None, 0, 1)
        bot.n_cut, bot.w_new = top.n_cut, top.w_new
        x = _Slab(case, law, dc, top, bot)
        taus = []
        for _ in range(S):
            x.step()
            taus.append(x.traction)
        tau = torch.stack(taus)
        (tau * bar).sum().backward()
        return tau.detach(), dc.grad
    X = _noalloc_input(case, seed).to(torch.complex128).reshape(case["n_lags"], 3, -1)
    hs = _HalfSpace(n1, n3, dx, case["n_lags"], 1, None, 0, case["n_lags"])
    Z = torch.zeros((4, 3, X.shape[2]), dtype=torch.complex128, device=DEV)
    for m in range(case["n_lags"]):
        Z += hs.w_new[:, hs.cls, m][:, None] * X[m]
    return hs.operator(Z, X[0]).reshape(3, n3, n1 // 2 + 1)
