"""The measured work: what programs have this library do, through its public
entry points (paper_1201_6062_gb300.tdse).

A case is one call of such a program on a synthetic hydrogen-like system
(energies and dipole blocks with the structure of inputs.py, drawn on the GPU):

  pulse     a window of a single pulse (Hamiltonian.propagate): RK4, truncated
            Taylor or short-iterative Lanczos, FP64 / float-float / FP32
            products, length or velocity gauge
  product   one Hamiltonian-vector product (Hamiltonian.hmatvec), the building
            block of a caller's own integrator
  batch     a window of many pulses on one Hamiltonian (propagate_batch)
  uneven    a window of several systems of different size (Group.propagate)
  adjoint   the gradient of a population with respect to every field sample
            (Hamiltonian.adjoint)
"""
import math

import numpy as np
import torch

from paper_1201_6062_gb300 import inputs, tdse

SCHEME_ORDER = {"rk4": 4, "taylor": 8, "lanczos": 10}
L2_BYTES = 129e6


def _pulse(prec, lmax, n, steps, scheme="rk4", gauge="length", sps=1, name=None):
    c = dict(kind="pulse", prec=prec, lmax=lmax, n=n, steps=steps, scheme=scheme, gauge=gauge, sps=sps)
    return dict(c, name=name) if name else c


def _batch(prec, lmax, n, pulses, steps, scheme="rk4", gauge="length", sps=1, name=None):
    c = dict(kind="batch", prec=prec, lmax=lmax, n=n, pulses=pulses, steps=steps, scheme=scheme, gauge=gauge, sps=sps)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the small workload (200 amplitudes, FP64 RK4): a parameter scan runs it again and
        # again, and each call is launch and latency bound
        _pulse("fp64", 3, 50, 100, name="small_pulse_fp64"),
        # one H x of a mid-size system, odd row length, as a caller's own integrator asks for
        dict(kind="product", prec="fp64", lmax=7, n=301, gauge="length", name="product_fp64"),
        # an L2-resident system between two read-outs, velocity gauge, Taylor series
        _pulse("df32", 15, 500, 20, scheme="taylor", gauge="velocity", name="mid_taylor_df32"),
        # the large single system (the benchmark's Hamiltonian) in FP64-class arithmetic
        _pulse("df32", 31, 2000, 8, name="large_rk4_df32"),
        # the same in plain FP64
        _pulse("fp64", 31, 2000, 2, name="large_rk4_fp64"),
        # the same with FP32 products and long Lanczos steps
        _pulse("fp32", 31, 2000, 2, scheme="lanczos", name="large_lanczos_fp32"),
        # the pulse sweep: 256 pulses on one Hamiltonian, fast products
        _batch("bf16x3", 15, 1000, 256, 4, name="sweep_bf16x3"),
        # the pulse sweep at FP64-class accuracy
        _batch("df32", 15, 1000, 256, 1, name="sweep_df32"),
        # a smaller sweep of ragged size, FP32 products, velocity gauge, Taylor series
        _batch("fp32", 9, 487, 100, 2, scheme="taylor", gauge="velocity", name="batch_fp32_odd"),
        # a handful of FP64 pulses on one Hamiltonian, samples on the half-step grid
        _batch("fp64", 7, 301, 24, 2, sps=2, name="batch_fp64_odd"),
        # systems of different (lmax, n) advanced together
        dict(kind="uneven", prec="df32", count=12, lmax_hi=20, n_hi=900, sizes=4, steps=4, name="uneven_df32"),
        # pulse shaping: the gradient with respect to every field sample
        dict(kind="adjoint", prec="fp64", lmax=15, n=500, steps=64, every=16, name="adjoint_fp64"),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _elems(case):
    return case["lmax"] * case["n"] ** 2


def draw(rng):
    kind = rng.choice(["pulse", "pulse", "product", "batch", "batch", "uneven", "adjoint"])
    gauge = rng.choice(["length", "velocity"])
    scheme = rng.choice(["rk4", "taylor"])
    sps = rng.choice([1, 2])
    while True:
        lmax, n = rng.randint(1, 31), _logint(rng, 20, 2000)
        if kind == "pulse":
            scheme = rng.choice(["rk4", "taylor", "lanczos"])
            c = _pulse(rng.choice(["fp64", "df32", "fp32"]), lmax, n, _logint(rng, 1, 40), scheme, gauge, sps)
            ok = _elems(c) * c["steps"] * SCHEME_ORDER[scheme] <= 4e9
        elif kind == "product":
            c = dict(kind="product", prec=rng.choice(["fp64", "df32", "fp32"]), lmax=lmax, n=n, gauge=gauge)
            ok = True
        elif kind == "batch":
            prec = rng.choice(["bf16x3", "df32", "fp32", "fp64"])
            pulses = _logint(rng, 2, 32 if prec == "fp64" else 256)
            c = _batch(prec, lmax, n, pulses, _logint(rng, 1, 8), scheme, gauge, sps)
            ok = (_elems(c) * c["steps"] * SCHEME_ORDER[scheme] * pulses <= (4e9 if prec == "fp64" else 1.6e10)
                  and _elems(c) <= 6e7)
        elif kind == "uneven":
            c = dict(kind="uneven", prec=rng.choice(["fp64", "df32", "fp32"]), count=rng.randint(2, 16),
                     lmax_hi=rng.randint(4, 20), n_hi=_logint(rng, 200, 900), sizes=rng.randint(0, 9999),
                     steps=_logint(rng, 1, 8))
            ok = True
        else:
            steps = _logint(rng, 4, 100)
            c = dict(kind="adjoint", prec=rng.choice(["fp64", "df32", "fp32"]), lmax=lmax, n=n, steps=steps,
                     every=rng.randint(1, steps))
            ok = _elems(c) * steps * 12 <= 4e9
        if ok:
            return c


# --------------------------------------------------------------- inputs --
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 1000003 + 17)


def _dipoles(lmax, n, gen):
    """Upper dipole blocks with N(0, 1)/sqrt(n) entries, on the GPU."""
    return torch.randn(lmax, n, n, dtype=torch.float64, device="cuda", generator=gen) / math.sqrt(n)


def _states(lmax, n, B, gen):
    """States in the middle of a pulse: most of the population still in the lowest level, the rest
    falling off with the angular momentum and with the energy of the continuum."""
    E = torch.from_numpy(inputs.energies(lmax, n)).cuda().reshape(lmax + 1, n)
    z = torch.randn(B, lmax + 1, n, 2, dtype=torch.float64, device="cuda", generator=gen)
    l = torch.arange(lmax + 1, dtype=torch.float64, device="cuda").reshape(-1, 1)
    c = torch.view_as_complex(z) * torch.exp(-0.3 * l) / (1.0 + E.abs()) ** 2
    c *= 0.3 / c.abs().square().sum((1, 2), keepdim=True).sqrt()
    c[:, 0, 0] += 0.9
    return c.reshape(B, -1).contiguous()


def _fields(count, dt, steps, sps, rng):
    """Windows of sin^2 pulses near their maximum: E0 log-uniform 0.01..0.1, omega 0.3..0.9."""
    out = []
    for _ in range(count):
        E0, om = math.exp(rng.uniform(math.log(0.01), math.log(0.1))), rng.uniform(0.3, 0.9)
        t0 = rng.uniform(0.4, 0.6) * inputs.pulse_duration(om)
        out.append(inputs.field_samples(E0, om, dt, steps, sps, t0=t0))
    return torch.from_numpy(np.stack(out)).cuda()


def _dt(case):
    # fixed-step schemes take dt 0.01, Taylor 8 and Lanczos the longer steps they are used for
    return {"rk4": 0.01, "taylor": 0.02, "lanczos": 0.05}[case.get("scheme", "rk4")]


def _members(case):
    """The sizes (lmax, n) of an uneven batch."""
    rng, lo = np.random.default_rng(case["sizes"]), min(100, case["n_hi"])
    return [(int(rng.integers(3, case["lmax_hi"] + 1)), int(rng.integers(lo, case["n_hi"] + 1)))
            for _ in range(case["count"])]


def _raw(case, seed):
    """The inputs alone: per system (lmax, n, dipole blocks), states and fields."""
    gen, rng = _gen(seed), np.random.default_rng(seed)
    if case["kind"] == "uneven":
        sysm = [(lm, n, _dipoles(lm, n, gen)) for lm, n in _members(case)]
        cs = [_states(lm, n, 1, gen)[0] for lm, n, _ in sysm]
        return sysm, cs, _fields(len(sysm), 0.01, case["steps"], 1, rng)
    lm, n = case["lmax"], case["n"]
    U = _dipoles(lm, n, gen)
    c = _states(lm, n, case.get("pulses", 1), gen)
    F = _fields(case.get("pulses", 1), _dt(case), case.get("steps", 1), case.get("sps", 1), rng)
    return [(lm, n, U)], c, F


def prepare(case, seed):
    sysm, c, F = _raw(case, seed)
    hams = [tdse.Hamiltonian(inputs.energies(lm, n), U.cpu().numpy(), lm, n, case["prec"]) for lm, n, U in sysm]
    if case.get("gauge", "length") != "length":
        hams[0].set_gauge(case["gauge"])
    st = dict(case=case, H=hams[0], F=F)
    if case["kind"] == "uneven":
        st.update(group=tdse.Group(hams), c0=c, c=[torch.empty_like(x) for x in c], F=list(F))
    elif case["kind"] == "adjoint":
        w = torch.from_numpy((inputs.energies(case["lmax"], case["n"]) < 0).astype(np.float64)).cuda()
        st.update(c0=c[0].contiguous(), F=F[0].contiguous(), w=w)
    elif case["kind"] == "batch":
        st.update(c0=c, c=torch.empty_like(c))
    else:
        st.update(c0=c[0].contiguous(), c=torch.empty_like(c[0]), F=F[0].contiguous())
    return st


def run(st):
    case, H = st["case"], st["H"]
    kind = case["kind"]
    if kind == "product":
        return H.hmatvec(st["c0"], 0.05, y=st["c"])
    if kind == "adjoint":
        grad, cT, loss = H.adjoint(st["c0"], st["F"], 0.01, case["steps"], st["w"], checkpoint_every=case["every"])
        return grad, torch.view_as_real(cT), loss
    if kind == "uneven":
        for c, c0 in zip(st["c"], st["c0"]):
            c.copy_(c0)
        return st["group"].propagate(st["c"], st["F"], 0.01, case["steps"])
    # the initial states are kept for the next run: the propagation works in place on a copy
    c = st["c"].copy_(st["c0"])
    kw = dict(scheme=case["scheme"], order=SCHEME_ORDER[case["scheme"]], samples_per_step=case["sps"])
    if kind == "batch":
        return H.propagate_batch(c, st["F"], case["pulses"], _dt(case), case["steps"], **kw)
    return H.propagate(c, st["F"], _dt(case), case["steps"], **kw)


# ------------------------------------------------------- work, tolerance --
def work(case):
    """Bytes: dipole blocks in the storage format of the precision, read once per call, or once per
    block product where they do not fit in L2; states and fields once in and once out.  Operations:
    8 per dipole element, pulse and product (row and column use, real and imaginary part, multiply and
    add), three times that for bf16x3, whose definition is three products."""
    kind, prec = case["kind"], case["prec"]
    eb = {"fp64": 8, "df32": 8, "fp32": 4, "bf16x3": 4}[prec]
    if kind == "uneven":
        elems = float(sum(lm * n * n for lm, n in _members(case)))
        amps = float(sum((lm + 1) * n for lm, n in _members(case)))
    else:
        elems, amps = float(_elems(case)), float((case["lmax"] + 1) * case["n"])
    steps, B = case.get("steps", 1), case.get("pulses", 1)
    products = {"product": 1, "adjoint": 12 * steps}.get(kind, steps * SCHEME_ORDER[case.get("scheme", "rk4")])
    ub = elems * eb
    sweeps = products if ub > L2_BYTES else 1
    io = amps * B * 32.0 + 8.0 * B * (case.get("sps", 1) * steps + 1)
    return {"bytes": ub * sweeps + io, "flops": 8.0 * elems * B * products * (3 if prec == "bf16x3" else 1)}


def tolerance(case):
    # about four times the distance from the 64-bit result measured on GB300 over these ranges
    rel = {"fp64": 1e-13, "df32": 1e-11, "fp32": 4e-6, "bf16x3": 4e-7}[case["prec"]]
    # most of a state's norm sits in its lowest level, so its root mean square is small beside that value
    return {"rel": rel, "max": 200 * rel}


# --------------------------------------------------- plain 64-bit result --
def _hx(E, U, x, f, velocity):
    """H x for x [L, n, K] (complex, K pulses) with fields f [K]: E x + f D x."""
    y = torch.zeros_like(x)
    if U.shape[0]:
        r = torch.view_as_real(x)
        n, K = x.shape[1], x.shape[2]
        up = torch.bmm(U, r[1:].reshape(-1, n, 2 * K)).reshape(-1, n, K, 2)
        dn = torch.bmm(U.transpose(1, 2), r[:-1].reshape(-1, n, 2 * K)).reshape(-1, n, K, 2)
        up, dn = torch.view_as_complex(up.contiguous()), torch.view_as_complex(dn.contiguous())
        if velocity:
            up, dn = 1j * up, -1j * dn
        y = torch.cat([up, torch.zeros_like(x[:1])]) + torch.cat([torch.zeros_like(x[:1]), dn])
    return E.unsqueeze(-1) * x + f * y


def _at(F, sps, k, h):
    """Fields [K] at t_k + h dt/2 from samples F [K, S]."""
    if sps == 2:
        return F[:, 2 * k + h]
    return F[:, k] if h == 0 else F[:, k + 1] if h == 2 else 0.5 * (F[:, k] + F[:, k + 1])


def _step(case, E, U, x, F, k, dt, velocity):
    sps, scheme = case.get("sps", 1), case.get("scheme", "rk4")
    g = lambda y, f: -1j * _hx(E, U, y, f, velocity)  # noqa: E731
    if scheme == "rk4":
        f0, fm, f1 = (_at(F, sps, k, h) for h in (0, 1, 2))
        k1 = g(x, f0)
        k2 = g(x + 0.5 * dt * k1, fm)
        k3 = g(x + 0.5 * dt * k2, fm)
        k4 = g(x + dt * k3, f1)
        return x + dt / 6.0 * (k1 + 2.0 * k2 + 2.0 * k3 + k4)
    f = _at(F, sps, k, 0)
    if scheme == "taylor":
        T, s = x, x
        for m in range(1, SCHEME_ORDER["taylor"] + 1):
            T = (dt / m) * g(T, f)
            s = s + T
        return s
    # short-iterative Lanczos: three-term recurrence, exponential of the tridiagonal matrix
    m, nrm = SCHEME_ORDER["lanczos"], torch.linalg.vector_norm(x)
    V, al, be = [x / nrm], [], []
    for j in range(m):
        w = _hx(E, U, V[j], f, velocity)
        al.append(torch.sum(V[j].conj() * w).real)
        w = w - al[j] * V[j] - (be[j - 1] * V[j - 1] if j else 0.0)
        be.append(torch.linalg.vector_norm(w))
        V.append(w / be[j])
    T = torch.diag(torch.stack(al)) + torch.diag(torch.stack(be[:-1]), 1) + torch.diag(torch.stack(be[:-1]), -1)
    ev, Q = torch.linalg.eigh(T.cpu())
    y = (Q.to(torch.complex128) * torch.exp(-1j * dt * ev)) @ Q[0].to(torch.complex128)
    return nrm * sum(y[j].item() * V[j] for j in range(m))


def _run_exact(case, lm, n, U, c, F, dt):
    """Final states [K, N] of the window from c [K, N] under F [K, S]."""
    E = torch.from_numpy(inputs.energies(lm, n)).cuda().reshape(lm + 1, n)
    velocity = case.get("gauge", "length") != "length"
    x = c.reshape(-1, lm + 1, n).permute(1, 2, 0)
    for k in range(case["steps"]):
        x = _step(case, E, U, x, F, k, dt, velocity)
    return x.permute(2, 0, 1).reshape(c.shape)


def exact(case, seed):
    sysm, c, F = _raw(case, seed)
    lm, n, U = sysm[0]
    kind = case["kind"]
    with torch.no_grad():
        if kind == "product":
            E = torch.from_numpy(inputs.energies(lm, n)).cuda().reshape(lm + 1, n)
            return _hx(E, U, c.reshape(lm + 1, n, 1), 0.05, case["gauge"] != "length").reshape(-1)
        if kind == "uneven":
            return [_run_exact(case, a, b, u, x.reshape(1, -1), f.reshape(1, -1), 0.01).reshape(-1)
                    for (a, b, u), x, f in zip(sysm, c, F)]
        if kind in ("pulse", "batch"):
            y = _run_exact(case, lm, n, U, c, F, _dt(case))
            return y if kind == "batch" else y.reshape(-1)
    F = F.clone().requires_grad_(True)
    w = torch.from_numpy((inputs.energies(lm, n) < 0).astype(np.float64)).cuda()
    y = _run_exact(case, lm, n, U, c, F, 0.01).reshape(-1)
    loss = torch.sum(w * (y.real ** 2 + y.imag ** 2))
    (grad,) = torch.autograd.grad(loss, F)
    return grad.reshape(-1), torch.view_as_real(y.detach()), loss.detach().reshape(1)
