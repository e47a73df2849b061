"""Workloads of the Dirac Lanczos library, as a user's program calls it, for measuring speed and accuracy.

`listed()` names them, `draw()` gives more of the same ranges, `prepare()` makes
what a program holds before the call (states, potentials, field schedules and
the propagator object with its workspace), `run()` is one pass through the
public entry points, `work()` the bytes and operations a pass cannot do
without, and `exact()` the same result in plain 64-bit torch/numpy.

A propagation advances its state in place, so a second pass on the same state
continues the packet, as a program's time loop does.
"""
import math

import numpy as np
import torch
import torch.utils.checkpoint

from paper_1407_7370_gb300.propagator import (BatchPropagator, Propagator, pulse_schedule,
                                               pulse_sine_basis_means)

C = 137.036
MC2 = C * C


def listed():
    return [
        # The smallest call: one step of the 64 x 64 free packet (m = 10), as in
        # a loop that looks at the state after every step.
        dict(name="step_64", kind="steps", precision="fp64", nx=64, ny=64, dx=0.1, m=10, steps=1, dt=1e-4,
             order=2, boundary="periodic", z=0.0, a0=0.0, ay=0.0),
        # The benchmark workload: a packet in a laser pulse, 1024 x 1024, m = 20.
        dict(name="laser_1024", kind="steps", precision="fp64", nx=1024, ny=1024, dx=0.05, m=20, steps=2, dt=2e-4,
             order=2, boundary="periodic", z=0.0, a0=50.0, ay=0.0),
        # The same workload on the mixed-precision path.
        dict(name="laser_1024_mixed", kind="steps", precision="mixed", nx=1024, ny=1024, dx=0.05, m=20, steps=2,
             dt=2e-4, order=2, boundary="periodic", z=0.0, a0=50.0, ay=0.0),
        # A packet passing an atom in a box: fourth-order stencil, Dirichlet
        # walls, a Coulomb potential, both vector-potential components, a ragged grid.
        dict(name="atom_301x203", kind="steps", precision="fp64", nx=301, ny=203, dx=0.08, m=16, steps=3, dt=1e-4,
             order=4, boundary="dirichlet", z=20.0, a0=30.0, ay=4.0),
        # A large free packet with m = 10 (the shape of the paper's own
        # benchmark, at 4096 x 4096 sites).
        dict(name="packet_4096", kind="steps", precision="fp64", nx=4096, ny=4096, dx=1e-3, m=10, steps=1, dt=1e-7,
             order=2, boundary="periodic", z=0.0, a0=0.0, ay=0.0),
        # Propagation of a state that lives in (pinned) host memory, copies
        # included, mixed precision, around a nucleus.
        dict(name="host_512_mixed", kind="host", precision="mixed", nx=512, ny=512, dx=0.05, m=16, steps=2, dt=1e-4,
             order=2, boundary="periodic", z=1.0, a0=20.0, ay=0.0),
        # A parameter scan on the mixed path: packets of different momenta and
        # laser amplitudes on grids of 128^2 .. 512^2.
        dict(name="batch_48_mixed", kind="batch", precision="mixed", n=48, side_lo=128, side_hi=512, side_step=128,
             dx=0.05, m=16, steps=2, dt=2e-4, order=2, boundary="periodic"),
        # A small FP64 scan on ragged grids.
        dict(name="batch_12", kind="batch", precision="fp64", n=12, side_lo=93, side_hi=301, side_step=1,
             dx=0.05, m=16, steps=2, dt=2e-4, order=2, boundary="periodic"),
        # H psi alone (energies, residuals) on the 2048 x 2048 Coulomb grid.
        dict(name="apply_2048", kind="apply", nx=2048, ny=2048, dx=0.02, order=2, boundary="periodic", z=20.0,
             a0=0.0, ay=0.0),
        # Bound states of a smoothed Coulomb potential, with full
        # reorthogonalisation; the lowest three (a doubler triplet).
        dict(name="eigs_1024", kind="eigs", nx=1024, ny=1024, dx=0.1, order=2, boundary="periodic", z=60.0,
             n_want=3, max_iter=160),
        # The same mode on a small ragged box, where launches and the checks count.
        dict(name="eigs_97x83", kind="eigs", nx=97, ny=83, dx=0.1, order=4, boundary="dirichlet", z=60.0,
             n_want=1, max_iter=160),
        # Gradient of a final-state observable with respect to the potential
        # (4 x 4 blocks) and the pulse coefficients.
        dict(name="adjoint_512", kind="adjoint", nx=512, ny=512, dx=0.05, m=16, steps=6, dt=2e-4, order=2,
             boundary="periodic", z=2.0, observable="px", block=4, n_coef=16, every=3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["steps", "steps", "steps", "steps", "batch", "batch", "apply", "eigs", "adjoint", "host"])
    order = rng.choice([2, 2, 2, 4])
    boundary = rng.choice(["periodic", "periodic", "dirichlet"])
    if kind in ("steps", "host"):
        nx, ny = _log_int(rng, 48, 2048), _log_int(rng, 48, 2048)
        return dict(kind=kind, precision=rng.choice(["fp64", "mixed"]), nx=nx, ny=ny, dx=rng.choice([0.05, 0.08, 0.1]),
                    m=rng.randint(8, 24), steps=rng.randint(1, 2), dt=rng.choice([1e-4, 5e-5, -1e-4]), order=order,
                    boundary=boundary, z=rng.choice([0.0, 0.0, 1.0, 20.0]), a0=rng.choice([0.0, 10.0, 50.0]),
                    ay=rng.choice([0.0, 0.0, 5.0]))
    if kind == "batch":
        hi = _log_int(rng, 96, 512)
        return dict(kind=kind, precision=rng.choice(["fp64", "mixed"]), n=_log_int(rng, 2, 40),
                    side_lo=max(32, hi // 4), side_hi=hi, side_step=rng.choice([1, 16]), dx=0.05,
                    m=rng.randint(8, 20), steps=2, dt=1e-4, order=order, boundary=boundary)
    if kind == "apply":
        return dict(kind=kind, nx=_log_int(rng, 64, 3000), ny=_log_int(rng, 64, 3000), dx=0.02, order=order,
                    boundary=boundary, z=rng.choice([0.0, 20.0]), a0=rng.choice([0.0, 10.0]), ay=0.0)
    if kind == "eigs":   # fourth order: the lowest state of Z = 60 is not degenerate
        return dict(kind=kind, nx=_log_int(rng, 96, 900), ny=_log_int(rng, 96, 900), dx=0.1, order=4,
                    boundary=boundary, z=60.0, n_want=1, max_iter=160)
    b = rng.choice([1, 2, 4])
    return dict(kind=kind, nx=b * _log_int(rng, 24, 120), ny=b * _log_int(rng, 24, 120), dx=0.05, m=rng.randint(12, 16),
                steps=rng.randint(2, 6), dt=1e-4, order=order, boundary=boundary, z=rng.choice([1.0, 5.0]),
                observable=rng.choice(["px", "proj"]), block=b, n_coef=rng.randint(2, 16), every=rng.randint(1, 4))


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------

def _dev():
    return torch.device("cuda") if torch.cuda.is_available() else torch.device("cpu")


def _packet(nx, ny, dx, p0, sigma, centre):
    """Gaussian superposition of positive-energy free states (mean momentum p0,
    width sigma, centred at `centre` from the middle of the grid), normalised
    to sum |psi|^2 dx^2 = 1; complex128 (ny, nx, 2)."""
    d = _dev()
    kx = (2 * math.pi * torch.fft.fftfreq(nx, d=dx, dtype=torch.float64, device=d))[None, :]
    ky = (2 * math.pi * torch.fft.fftfreq(ny, d=dx, dtype=torch.float64, device=d))[:, None]
    e = torch.sqrt(MC2 * MC2 + MC2 * (kx * kx + ky * ky))
    amp = torch.exp(-((kx - p0[0]) ** 2 + (ky - p0[1]) ** 2) * sigma ** 2) / torch.sqrt(2 * e * (e + MC2))
    phase = kx * ((nx // 2) * dx + centre[0]) + ky * ((ny // 2) * dx + centre[1])
    amp = torch.polar(amp, -phase)
    psi = torch.empty((ny, nx, 2), dtype=torch.complex128, device=d)
    psi[..., 0] = torch.fft.ifft2(amp * (e + MC2))
    psi[..., 1] = torch.fft.ifft2(amp * C * torch.complex(kx.expand(ny, nx), ky.expand(ny, nx)))
    return psi / math.sqrt(float((psi.abs() ** 2).sum()) * dx * dx)


def _coords(nx, ny, dx):
    d = _dev()
    x = (torch.arange(nx, dtype=torch.float64, device=d) - nx // 2) * dx
    y = (torch.arange(ny, dtype=torch.float64, device=d) - ny // 2) * dx
    return x[None, :], y[:, None]


def _coulomb(nx, ny, dx, z, off):
    x, y = _coords(nx, ny, dx)
    return (-z / torch.sqrt((x - off[0]) ** 2 + (y - off[1]) ** 2 + 0.25)).contiguous()


def _random_packet(c, rng, p_max=None):
    nx, ny, dx = c["nx"], c["ny"], c["dx"]
    box = dx * min(nx, ny)
    sigma = min(1.0, box / 10.0) * rng.uniform(0.9, 1.1)
    p = rng.uniform(0.5, 1.0) * (p_max if p_max is not None else min(20.0, 1.0 / dx))
    th = rng.uniform(-math.pi, math.pi)
    centre = (rng.uniform(-0.05, 0.05) * box, rng.uniform(-0.05, 0.05) * box)
    return _packet(nx, ny, dx, (p * math.cos(th), p * math.sin(th)), sigma, centre)


def _schedule(c, rng, a0, ay, n):
    """(n, 2) step means of A in the middle of a sin^2 pulse of one atomic unit."""
    dt = abs(c["dt"])
    A = pulse_schedule(rng.uniform(0.3, 0.6), dt, n, a0, 0.05, 1.0)
    if ay:
        A[:, 1] = ay * rng.uniform(0.5, 1.0, size=n)
    return A


def _inputs(c, seed):
    rng = np.random.default_rng(seed)
    k = c["kind"]
    if k in ("steps", "host"):
        psi = _random_packet(c, rng, 100.0 if c["dx"] < 0.01 else None)
        off = rng.uniform(-0.3, 0.3, size=2)
        V = _coulomb(c["nx"], c["ny"], c["dx"], c["z"], off) if c["z"] else None
        A = _schedule(c, rng, c["a0"], c["ay"], c["steps"]) if c["a0"] or c["ay"] else None
        return dict(psi=psi, V=V, A=A, shift=MC2 if c["precision"] == "mixed" else 0.0)
    if k == "batch":
        # the sizes belong to the case, the packets and fields to the seed
        sizes = np.random.default_rng(c["n"] * 1000 + c["side_hi"])
        lo, hi, st = c["side_lo"], c["side_hi"], c["side_step"]
        ns = [int(s) for s in lo + st * sizes.integers(0, (hi - lo) // st + 1, size=c["n"])]
        grids = [(s, s, c["dx"], c["dx"]) for s in ns]
        flat = torch.empty((sum(s * s for s in ns), 2), dtype=torch.complex128, device=_dev())
        psis, at = [], 0
        for s in ns:
            box = s * c["dx"]
            v = flat[at:at + s * s].view(s, s, 2)
            v.copy_(_packet(s, s, c["dx"], (rng.uniform(0.0, 50.0), 0.0), min(1.0, box / 10.0), (0.0, 0.0)))
            psis.append(v)
            at += s * s
        A = np.stack([_schedule(c, rng, rng.uniform(0.0, 100.0), 0.0, c["steps"]) for _ in ns], axis=1)
        return dict(flat=flat, psis=psis, grids=grids, A=A, shift=MC2 if c["precision"] == "mixed" else 0.0)
    if k == "apply":
        psi = _random_packet(c, rng)
        V = _coulomb(c["nx"], c["ny"], c["dx"], c["z"], rng.uniform(-0.3, 0.3, size=2)) if c["z"] else None
        return dict(psi=psi, V=V, A=(c["a0"], c["ay"]), shift=MC2)
    if k == "eigs":
        x, y = _coords(c["nx"], c["ny"], c["dx"])
        w, a, b = rng.uniform(0.8, 1.2), rng.uniform(0.2, 0.4), rng.uniform(0.1, 0.3)
        s = torch.zeros((c["ny"], c["nx"], 2), dtype=torch.complex128, device=_dev())
        s[..., 0] = torch.exp(-(x * x + y * y) * w) * (1 + a * x + b * y)
        return dict(start=s, V=_coulomb(c["nx"], c["ny"], c["dx"], c["z"], (0.0, 0.0)), shift=MC2)
    psi = _random_packet(c, rng)
    V = _coulomb(c["nx"], c["ny"], c["dx"], c["z"], rng.uniform(-0.3, 0.3, size=2))
    W = pulse_sine_basis_means(c["steps"], c["dt"], c["n_coef"], c["steps"] * c["dt"])
    A = np.zeros((c["steps"], 2))
    A[:, 0] = W @ rng.normal(0.0, 10.0, size=c["n_coef"])
    phi = _random_packet(c, rng) if c["observable"] == "proj" else None
    if phi is not None:
        phi = 0.6 * phi + 0.8 * psi
    return dict(psi0=psi, V=V, W=W, A=A, phi=phi, shift=0.0)


def _propagator(c, m, precision="fp64"):
    return Propagator(c["nx"], c["ny"], c["dx"], c["dx"], order=c["order"], boundary=c["boundary"], m_max=m,
                      precision=precision)


def prepare(case, seed):
    c, s = case, _inputs(case, seed)
    s["case"] = c
    k = c["kind"]
    if k in ("steps", "host"):
        p = _propagator(c, c["m"], c["precision"])
        p.set_fields(s["V"], shift=s["shift"])
        if k == "host":
            s["psi"] = s["psi"].cpu().pin_memory()
    elif k == "batch":
        p = BatchPropagator(s["grids"], order=c["order"], boundary=c["boundary"], m_max=c["m"], precision=c["precision"])
        for b in range(p.n):
            p.set_fields(b, None, shift=s["shift"])
    elif k == "apply":
        p = _propagator(c, 1)
        p.set_fields(s["V"], A=s["A"], shift=s["shift"])
        s["out"] = torch.empty_like(s["psi"])
    elif k == "eigs":
        p = _propagator(c, 1)
        p.set_fields(s["V"], shift=s["shift"])
    else:
        p = _propagator(c, c["m"])
        p.set_fields(s["V"], shift=s["shift"])
    s["prop"] = p
    return s


def run(state):
    c, p = state["case"], state["prop"]
    k = c["kind"]
    if k == "steps":
        p.steps(state["psi"], c["steps"], c["dt"], c["m"], A=state["A"])
        return state["psi"]
    if k == "host":
        p.propagate_host(state["psi"], c["steps"], c["dt"], c["m"], A=state["A"])
        return state["psi"]
    if k == "batch":
        p.steps(state["psis"], c["steps"], c["dt"], c["m"], A=state["A"])
        return state["flat"]
    if k == "apply":
        return p.apply(state["psi"], state["out"])
    if k == "eigs":
        r = p.eigs(state["start"], n_want=c["n_want"], max_iter=c["max_iter"], tol=1e-8, window=(-MC2, 0.0))
        return {"values": r.values}
    r = p.adjoint_gradient(state["psi0"], c["steps"], c["dt"], c["m"], state["A"], observable=c["observable"],
                           phi=state["phi"], checkpoint_every=c["every"], block=(c["block"], c["block"]),
                           W=state["W"], return_state=True)
    return {"loss": r.loss, "dV": r.dV, "dA": r.dA, "da": r.da, "psiN": r.psiN}


def work(case):
    """A Lanczos step of m vectors takes 96 m operations a site (80 for each
    product with its sums, 16 for each recombined vector); its state is read
    and written once.  An eigen iteration reads every earlier vector."""
    c = case
    k = c["kind"]
    if k == "batch":
        sizes = np.random.default_rng(c["n"] * 1000 + c["side_hi"])
        ns = c["side_lo"] + c["side_step"] * sizes.integers(0, (c["side_hi"] - c["side_lo"]) // c["side_step"] + 1,
                                                            size=c["n"])
        n = float(sum(int(s) * int(s) for s in ns))
    else:
        n = float(c["nx"] * c["ny"])
    v = 8.0 * n if c.get("z") else 0.0
    if k in ("steps", "host", "batch"):
        return {"bytes": 64.0 * n + v, "flops": 96.0 * c["m"] * c["steps"] * n}
    if k == "apply":
        return {"bytes": 64.0 * n + v, "flops": 44.0 * n}
    if k == "eigs":
        it = 100.0   # about where the wanted values converge
        return {"bytes": 32.0 * n * it * it / 2, "flops": 64.0 * n * it * it / 2}
    # forward, the recomputed segment, and the two Krylov spaces of every
    # backward step, then the contraction of the two bases
    return {"bytes": 72.0 * n, "flops": c["steps"] * n * (4 * 96.0 * c["m"] + 16.0 * c["m"] ** 2)}


# ----------------------------------------------------------------------------
# the same results in plain 64-bit torch / numpy
# ----------------------------------------------------------------------------

def _shifted(f, dim, o, dirichlet):
    g = torch.roll(f, -o, dims=dim)
    if dirichlet:
        n = f.shape[dim]
        keep = torch.arange(n, device=f.device)
        keep = ((keep + o >= 0) & (keep + o < n)).to(torch.float64)
        g = g * (keep[:, None, None] if dim == 0 else keep[None, :, None])
    return g


def _diff(f, dim, h, order, dirichlet):
    d1 = _shifted(f, dim, 1, dirichlet) - _shifted(f, dim, -1, dirichlet)
    if order == 2:
        return d1 / (2 * h)
    return (8 * d1 - (_shifted(f, dim, 2, dirichlet) - _shifted(f, dim, -2, dirichlet))) / (12 * h)


def _h(f, dx, order, boundary, V, ax, ay, shift):
    """(H - shift) f."""
    d = boundary == "dirichlet"
    px = -1j * _diff(f, 1, dx, order, d) + ax * f
    py = -1j * _diff(f, 0, dx, order, d) + ay * f
    v = (V if V is not None else 0.0) - shift
    up = (MC2 + v) * f[..., 0] + C * (px[..., 1] - 1j * py[..., 1])
    lo = (-MC2 + v) * f[..., 1] + C * (px[..., 0] + 1j * py[..., 0])
    return torch.stack((up, lo), dim=-1)


def _lanczos_step(psi, apply, dt, m, shift):
    nrm = float(torch.linalg.vector_norm(psi))
    q, al, be = [psi / nrm], [], []
    for i in range(m):
        z = apply(q[i])
        if i:
            z = z - be[-1] * q[i - 1]
        al.append(float(torch.vdot(q[i].reshape(-1), z.reshape(-1)).real))
        if i + 1 == m:
            break
        z = z - al[-1] * q[i]
        be.append(float(torch.linalg.vector_norm(z)))
        q.append(z / be[-1])
    lam, S = np.linalg.eigh(np.diag(al) + np.diag(be, 1) + np.diag(be, -1))
    v = nrm * np.exp(-1j * shift * dt) * (S @ (np.exp(-1j * lam * dt) * S[0]))
    out = torch.zeros_like(psi)
    for j in range(m):
        out += complex(v[j]) * q[j]
    return out


def _propagated(c, psi, dx, V, A, n):
    for k in range(n):
        ax, ay = (float(A[k][0]), float(A[k][1])) if A is not None else (0.0, 0.0)
        # energies from m c^2 (where the packets are): less cancellation
        psi = _lanczos_step(psi, lambda f: _h(f, dx, c["order"], c["boundary"], V, ax, ay, MC2), c["dt"], c["m"], MC2)
    return psi


def _exact_eigs(c, s):
    n = c["nx"] * c["ny"] * 2
    Q = torch.empty((c["max_iter"] + 1, n), dtype=torch.complex128, device=_dev())
    v = s["start"].reshape(-1)
    Q[0] = v / torch.linalg.vector_norm(v)
    al, be = [], []
    for i in range(c["max_iter"]):
        z = _h(Q[i].view(c["ny"], c["nx"], 2), c["dx"], c["order"], c["boundary"], s["V"], 0.0, 0.0, MC2).reshape(-1)
        a = 0.0
        for _ in range(2):
            h = torch.mv(Q[:i + 1].conj(), z)
            z = z - torch.mv(Q[:i + 1].T, h)
            a += float(h[i].real)
        al.append(a)
        be.append(float(torch.linalg.vector_norm(z)))
        Q[i + 1] = z / be[-1]
        if (i + 1) % 10 == 0:
            th, S = np.linalg.eigh(np.diag(al) + np.diag(be[:-1], 1) + np.diag(be[:-1], -1))
            bound = np.abs(be[-1] * S[-1])
            ok = (bound <= 1e-8 * np.maximum(1.0, np.abs(th))) & (th > -MC2) & (th < 0)
            if ok.sum() >= c["n_want"]:
                return {"values": th[ok][:c["n_want"]]}
    return None


def _exact_adjoint(c, s):
    """Reverse-mode differentiation of the propagation itself, each step's
    exponential as its Taylor series (to rounding)."""
    V = s["V"].clone().requires_grad_(True)
    A = torch.tensor(s["A"], dtype=torch.float64, device=_dev(), requires_grad=True)
    d = c["boundary"] == "dirichlet"

    def step(psi, V, a):
        term, out = psi, psi
        for k in range(1, 44):
            term = _h(term, c["dx"], c["order"], c["boundary"], V, a[0], a[1], 0.0) * (-1j * c["dt"] / k)
            out = out + term
        return out

    psi = s["psi0"]
    for n in range(c["steps"]):
        psi = torch.utils.checkpoint.checkpoint(step, psi, V, A[n], use_reentrant=False)
    w = c["dx"] * c["dx"]
    if c["observable"] == "px":
        loss = w * (psi.conj() * (-1j) * _diff(psi, 1, c["dx"], c["order"], d)).sum().real
    else:
        loss = (w * (s["phi"].conj() * psi).sum()).abs() ** 2
    loss.backward()
    b = c["block"]
    dA = A.grad.cpu().numpy()
    return {"loss": float(loss.detach()), "dV": V.grad.view(c["ny"] // b, b, c["nx"] // b, b).sum(dim=(1, 3)), "dA": dA,
            "da": s["W"].T @ dA[:, 0], "psiN": psi.detach()}


def exact(case, seed):
    c, s = case, _inputs(case, seed)
    k = c["kind"]
    if k in ("steps", "host"):
        return _propagated(c, s["psi"], c["dx"], s["V"], s["A"], c["steps"])
    if k == "batch":
        return torch.cat([_propagated(c, psi, c["dx"], None, s["A"][:, b], c["steps"]).reshape(-1, 2)
                          for b, psi in enumerate(s["psis"])])
    if k == "apply":
        return _h(s["psi"], c["dx"], c["order"], c["boundary"], s["V"], c["a0"], c["ay"], MC2)
    if k == "eigs":
        return _exact_eigs(c, s)
    return _exact_adjoint(c, s)
