"""What a user of this solver has it do, as cases to time.

A case is a dict of plain values with a "kind":

* "run": a Solver that holds its state on the GPU.  One pass advances the state by `steps` time steps and copies
  the state out to a device buffer, as a program does between two snapshots; with `observe` it reads the
  observables too (a relaxation that prints its energy).  The state goes on from pass to pass.
* "sweep": a Batch of independent 2D problems, advanced by `steps` steps, the states read back at the end.
* "gradient": the fidelity and its gradient through `steps` time steps (checkpoints every `every`).
* "potential": the dipolar potential of a caller's device state into a caller's buffer, without allocations.

Grids, spacings, couplings and time steps are those of the workloads in bench.py and of the tests, and of the
same order in draw().  All inputs are made from the seed.
"""
import math

import numpy as np
import torch

from paper_1601_04640_gb300 import dgpe, synth

KERNELS = {"dipolar3d": dgpe.DGPE_KERNEL_DIPOLAR_3D, "xy": dgpe.DGPE_KERNEL_QUASI2D_XY,
           "xz": dgpe.DGPE_KERNEL_QUASI2D_XZ}
# every supported line length: 2^k, 3 2^k and 5 2^k from 32 to 512
LENGTHS = [32, 40, 48, 64, 80, 96, 128, 160, 192, 256, 320, 384, 512]
QD = 0.5  # width of the transverse profile of the quasi-2D kernels


def _run(name, n, h, nu, g, gdd, dt, steps, fp64, imag, kernel="dipolar3d", split="lie", real=False, observe=False):
    n, h, nu = list(n) + [1] * (3 - len(n)), list(h) + [1.0] * (3 - len(h)), list(nu) + [0.0] * (3 - len(nu))
    return {"name": name, "kind": "run", "kernel": kernel, "nx": n[0], "ny": n[1], "nz": n[2], "hx": h[0], "hy": h[1],
            "hz": h[2], "nux": nu[0], "nuy": nu[1], "nuz": nu[2], "g": g, "gdd": gdd, "dt": dt, "steps": steps,
            "fp64": fp64, "imag": imag, "split": split, "real": real, "observe": observe}


def listed():
    return [
        # a small ground state in double precision, energy printed every 50 steps: launches and latency count
        _run("imag 32^3 fp64", (32,) * 3, (0.25,) * 3, (1.0, 1.0, 2.0), 50.0, 15.0, 2e-3, 50, True, True, observe=True),
        # the same size in single precision, in real time
        _run("real 32x64x48 fp32", (32, 64, 48), (0.25, 0.2, 0.3), (1.0, 1.3, 0.8), 50.0, 15.0, 2e-3, 50, False, False),
        # dynamics in a plane with the dipoles in it
        _run("xz 512^2 fp32", (512, 512), (0.05,) * 2, (1.0, 2.0), 150.0, 60.0, 5e-4, 50, False, False, "xz"),
        # a ground state in the plane on a grid that is no power of two, double precision
        _run("xy 96x160 fp64", (96, 160), (0.2, 0.15), (1.0, 1.5), 50.0, 20.0, 1e-3, 50, True, True, "xy", observe=True),
        # the headline workload, both precisions: quench dynamics of a cigar
        _run("real 256^3 fp32", (256,) * 3, (0.1,) * 3, (1.0, 1.0, 0.5), 150.0, 60.0, 5e-4, 10, False, False),
        _run("real 256^3 fp64", (256,) * 3, (0.1,) * 3, (1.0, 1.0, 0.5), 150.0, 60.0, 5e-4, 2, True, False),
        # its ground state with a real field
        _run("imag 256^3 fp32 real state", (256,) * 3, (0.1,) * 3, (1.0, 1.0, 0.5), 200.0, 60.0, 2e-3, 10, False, True,
             real=True, observe=True),
        # second-order dynamics on a box whose sides are 3 2^k, 5 2^k and 2^k
        _run("real 192x160x128 fp32 strang", (192, 160, 128), (0.12, 0.15, 0.18), (1.0, 1.2, 0.7), 150.0, 60.0, 1e-3, 10,
             False, False, split="strang"),
        # the largest grid: a pancake
        _run("real 512x512x256 fp32", (512, 512, 256), (0.08,) * 3, (1.0, 1.0, 3.0), 500.0, 200.0, 2e-4, 3, False, False),
        # a parameter sweep over uneven planes, half in imaginary and half in real time
        {"name": "sweep of 48 planes", "kind": "sweep", "count": 48, "params": 4640, "steps": 100},
        # optimal control: gradient of the fidelity with respect to g and eight modulation coefficients
        {"name": "gradient 128^3 fp32", "kind": "gradient", "nx": 128, "ny": 128, "nz": 128, "h": 0.15, "g": 200.0,
         "gdd": 60.0, "dt": 1e-3, "steps": 32, "every": 8, "fp64": False},
        # the potential alone, from another program's loop
        {"name": "potential 64^3 fp32", "kind": "potential", "kernel": "dipolar3d", "nx": 64, "ny": 64, "nz": 64,
         "h": 0.2, "fp64": False},
    ]


def draw(rng):
    kind = rng.choice(["run"] * 7 + ["sweep", "gradient", "potential"])
    if kind == "sweep":
        return {"kind": kind, "count": rng.randint(3, 48), "params": rng.randrange(1 << 30), "steps": rng.randint(20, 100)}
    if kind == "gradient":
        fp64 = rng.random() < 0.3
        n = [rng.choice([32, 48, 64, 80, 96, 128]) for _ in range(3)]
        return {"kind": kind, "nx": n[0], "ny": n[1], "nz": n[2], "h": rng.uniform(0.12, 0.3), "g": rng.uniform(50.0, 200.0),
                "gdd": rng.uniform(10.0, 60.0), "dt": _log(rng, 5e-4, 4e-3), "steps": rng.randint(8, 32),
                "every": rng.randint(3, 12), "fp64": fp64}
    if kind == "potential":
        plane = rng.random() < 0.5
        while True:
            n = [rng.choice([32, 64, 128, 256, 512]) for _ in range(2 if plane else 3)] + [1] * plane
            if n[0] * n[1] * n[2] <= 1 << 18:
                break
        return {"kind": kind, "kernel": "xy" if plane else "dipolar3d", "nx": n[0], "ny": n[1], "nz": n[2],
                "h": rng.uniform(0.05, 0.3), "fp64": rng.random() < 0.5}
    fp64, imag, dim = rng.random() < 0.4, rng.random() < 0.5, rng.choice([2, 3, 3])
    most = 1 << (22 if fp64 else 24)
    target = _log(rng, 1 << 12, most)  # sites, spread over their logarithm
    while True:
        n = [rng.choice(LENGTHS) for _ in range(dim)]
        if 0.5 < math.prod(n) / target < 2.0 or dim == 2 and target > 1 << 18:
            break
        target = target if rng.random() < 0.98 else _log(rng, 1 << 12, most)
    # a box some 8 to 25 trap lengths wide; tau = dt / (4 h^2) between about 0.002 and 0.4
    h = [min(0.3, max(0.05, rng.uniform(8.0, 25.0) / k)) for k in n]
    nu = [1.0] + [rng.uniform(0.5, 2.0) for _ in range(dim - 1)]
    g = rng.uniform(10.0, 200.0)
    c = _run("", n, h, nu, g, g * rng.uniform(0.05, 0.24), _log(rng, 2e-4, 4e-3),
             max(2, min(50, int(3e7 / math.prod(n) / (12 if fp64 else 1)))), fp64, imag,
             "dipolar3d" if dim == 3 else rng.choice(["xy", "xz"]), "lie" if imag or rng.random() < 0.8 else "strang",
             imag and rng.random() < 0.3, rng.random() < 0.4)
    del c["name"]
    return c


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


# ------------------------------------------------------------------ inputs
def _axes(case):
    """Sizes, spacings and trap frequencies, x first."""
    dim = 2 if case.get("kernel") in ("xy", "xz") else 3
    n = [case["nx"], case["ny"], case["nz"]][:dim]
    if "h" in case:
        return n, [case["h"]] * dim, [1.0, 1.0, 0.5][:dim]
    return n, [case["hx"], case["hy"], case["hz"]][:dim], [case["nux"], case["nuy"], case["nuz"]][:dim]


def _grid(n, h):
    """Coordinates (i - n/2) h of each axis, shaped to broadcast over [z][y][x]."""
    dim = len(n)
    return [((torch.arange(n[a], device="cuda", dtype=torch.float64) - n[a] // 2) * h[a])
            .reshape([n[a] if dim - 1 - a == d else 1 for d in range(dim)]) for a in range(dim)]


def _state(n, h, width, seed, noise=0.01):
    """A Gaussian of the given widths with 1 % complex noise, complex128 on the GPU."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    env = 1.0
    for x, a in zip(_grid(n, h), width):
        env = env * ((a / math.pi) ** 0.25 * torch.exp(-0.5 * a * x * x))
    shape = tuple(reversed(n))
    xi = torch.randn(shape + (2,), generator=gen, device="cuda", dtype=torch.float64)
    return env * (1.0 + noise * torch.view_as_complex(xi))


def _dtype(case):
    return torch.complex128 if case["fp64"] else torch.complex64


def _run_state(case, seed):
    n, h, nu = _axes(case)
    psi = _state(n, h, nu, seed)
    if case["real"]:
        psi = psi.real.to(psi.dtype)
    return psi.to(_dtype(case))


def _sweep(case, seed):
    """The problems of a sweep and the seeds of their states.  The dipoles are kept below the strength at which a
    plane is unstable at short wavelengths, where two computations of the same steps part by themselves."""
    problems = [dict(q, gdd=0.3 * q["gdd"]) for q in synth.batched_problems(case["params"], case["count"])]
    return problems, [seed * 1000 + i for i in range(len(problems))]


def _gradient_states(case, seed):
    """Start, target and modulation coefficients; host arrays, as the call takes them."""
    n, h, nu = _axes(case)
    psi0, target = _state(n, h, nu, 2 * seed), _state(n, h, [1.1, 0.9, 0.5], 2 * seed + 1)
    return psi0, target, [float(c) for c in synth.trap_modulation(160104640 + seed, 8)]


# ------------------------------------------------------------------ passes
def prepare(case, seed):
    kind = case["kind"]
    if kind == "sweep":
        problems, seeds = _sweep(case, seed)
        b = dgpe.Batch(problems)
        for i, (q, s) in enumerate(zip(problems, seeds)):
            b.set_psi(i, _state(q["n"], q["h"], q["nu"], s).cpu().numpy())
        return {"case": case, "batch": b}
    n, h, nu = _axes(case)
    if kind == "potential":
        psi = _state(n, h, nu, seed).to(_dtype(case))
        return {"case": case, "n": n, "h": h, "psi": psi, "phi": torch.empty(psi.shape, dtype=psi.real.dtype, device="cuda")}
    if kind == "gradient":
        psi0, target, cm = _gradient_states(case, seed)
        s = dgpe.Solver(3, n, h, nu, case["g"], case["gdd"], case["dt"], False, case["fp64"])
        s.set_trap_modulation(cm)
        return {"case": case, "solver": s, "psi0": psi0.cpu().numpy(), "target": target.cpu().numpy(), "M": len(cm)}
    s = dgpe.Solver(len(n), n, h, nu, case["g"], case["gdd"], case["dt"], case["imag"], case["fp64"], KERNELS[case["kernel"]],
                    QD, split=case["split"], real_psi=case["real"])
    psi = _run_state(case, seed)
    dgpe.dgpe_set_psi_device(s.h, psi.data_ptr(), psi.numel(), case["fp64"])
    return {"case": case, "solver": s, "out": torch.empty_like(psi)}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "sweep":
        b = state["batch"]
        b.step(case["steps"])
        # the states are held in single precision: kept so
        return {"psi": [b.get_psi(i).astype(np.complex64) for i in range(case["count"])]}
    if kind == "potential":
        dgpe.dgpe_dipolar_potential_noalloc(state["psi"].data_ptr(), state["phi"].data_ptr(), case["fp64"], len(state["n"]),
                                            state["n"], state["h"], KERNELS[case["kernel"]], QD,
                                            torch.cuda.current_stream().cuda_stream)
        return state["phi"]
    s = state["solver"]
    if kind == "gradient":
        f, dg, dc = dgpe.dgpe_fidelity_gradient(s.h, state["psi0"], state["target"], case["steps"], case["every"], state["M"])
        return {"F": f, "dg": dg, "dc": dc}
    out = state["out"]
    s.step(case["steps"])
    dgpe.dgpe_get_psi_device(s.h, out.data_ptr(), out.numel(), case["fp64"])
    got = {"psi": out}
    if case["observe"]:
        o = s.observables()
        got.update({k: o[k] for k in ("norm", "mu", "energy", "kin", "pot", "contact", "dipolar", "rms_r")})
    return got


def work(case):
    """The state is read and written once in a step; the operations are those of the transforms (5 N log2 N for a
    complex line of N, real data half), of the exponential (36 per site) and of the tridiagonal solves (28 per site
    and axis, complex)."""
    if case["kind"] == "sweep":
        n = [q["n"][0] for q in synth.batched_problems(case["params"], case["count"])]
        sites, lg, dim, steps, b = sum(k * k for k in n), 2 * math.log2(sum(n) / len(n)), 2, case["steps"], 8
        return {"bytes": 2.0 * b * sites * steps, "flops": sites * steps * (5.0 * lg + 36 + 28 * dim)}
    n, _, _ = _axes(case)
    sites, lg, b = math.prod(n), math.log2(math.prod(n)), 16 if case["fp64"] else 8
    convolve = 5.0 * lg + 5
    if case["kind"] == "potential":
        return {"bytes": 1.5 * b * sites, "flops": sites * convolve}
    step = convolve + 36 + 28 * len(n)
    if case["kind"] == "gradient":  # forward, the segments again, and the reverse step with two convolutions
        return {"bytes": 6.0 * b * sites * case["steps"], "flops": sites * case["steps"] * (3 * step + convolve)}
    b = b / 2 if case["real"] else b
    return {"bytes": 2.0 * b * sites * case["steps"], "flops": sites * case["steps"] * step}


# ---------------------------------------------------- the same in 64 bits
def _kernel_table(n, h, kernel):
    """U(k) over the full grid [z][y][x] (the second axis of "xz" is z)."""
    dim = len(n)
    q = [(2.0 * math.pi * torch.fft.fftfreq(n[a], h[a], device="cuda", dtype=torch.float64))
         .reshape([n[a] if dim - 1 - a == d else 1 for d in range(dim)]) for a in range(dim)]
    k2 = sum(x * x for x in q)
    if kernel == "dipolar3d":
        u = (4.0 * math.pi / 3.0) * (3.0 * q[2] ** 2 / torch.where(k2 > 0, k2, torch.ones_like(k2)) - 1.0)
        return torch.where(k2 > 0, u, torch.zeros_like(u))
    k = torch.sqrt(k2)
    e = torch.special.erfcx(k * QD / math.sqrt(2.0))
    pref = (4.0 * math.pi / 3.0) / (math.sqrt(2.0 * math.pi) * QD)
    if kernel == "xy":
        return pref * (2.0 - 3.0 * math.sqrt(math.pi / 2.0) * k * QD * e)
    kz2 = q[1] ** 2 / torch.where(k > 0, k, torch.ones_like(k))
    return pref * (3.0 * math.sqrt(math.pi / 2.0) * kz2 * QD * e - 1.0)


class _Exact:
    """The time step in complex128: Fourier transforms and dense Crank-Nicolson matrices."""

    def __init__(self, n, h, nu, gdd, dt, imag, kernel):
        self.n, self.h, self.gdd, self.dt, self.imag = n, h, gdd, dt, imag
        self.u = _kernel_table(n, h, kernel)
        self.v = sum(0.5 * w * w * x * x for w, x in zip(nu, _grid(n, h)))
        self.cn = []
        for k, d in zip(n, h):
            one = torch.eye(k, device="cuda", dtype=torch.complex128)
            off = torch.ones(k - 1, device="cuda", dtype=torch.complex128)
            t = 2.0 * one - torch.diag(off, 1) - torch.diag(off, -1)
            kt = (1.0 if imag else 1j) * dt / (4.0 * d * d)
            self.cn.append(torch.linalg.solve(one + kt * t, one - kt * t))

    def potential(self, density):
        return torch.fft.ifftn(self.u * torch.fft.fftn(density.to(torch.complex128))).real

    def kick(self, psi, g, s, dt):
        n = psi.real ** 2 + psi.imag ** 2
        th = dt * (s * self.v + g * n + self.gdd * self.potential(n))
        return psi * (torch.exp(-th) if self.imag else torch.exp(-1j * th))

    def kinetic(self, psi):
        shape = psi.shape
        psi = (psi.reshape(-1, shape[-1]) @ self.cn[0].T).reshape(shape)
        psi = self.cn[1] @ psi
        if len(shape) == 3:
            psi = (self.cn[2] @ psi.reshape(shape[0], -1)).reshape(shape)
        return psi

    def step(self, psi, g, s=1.0, strang=False):
        psi = self.kinetic(self.kick(psi, g, s, self.dt / 2 if strang else self.dt))
        if strang:
            psi = self.kick(psi, g, s, self.dt / 2)
        if self.imag:
            psi = psi / torch.sqrt(math.prod(self.h) * (psi.real ** 2 + psi.imag ** 2).sum())
        return psi

    def observe(self, psi, g):
        cell, n = math.prod(self.h), psi.real ** 2 + psi.imag ** 2
        norm = cell * n.sum()
        kin = 0.0
        for a, d in enumerate(self.h):
            axis = psi.dim() - 1 - a
            edge = torch.zeros_like(psi.narrow(axis, 0, 1))
            kin = kin + (torch.diff(psi, dim=axis, prepend=edge, append=edge).abs() ** 2).sum() / (2.0 * d * d)
        kin = cell * kin / norm
        pot = cell * (self.v * n).sum() / norm
        contact = g * cell * (n * n).sum() / norm
        dipolar = self.gdd * cell * (self.potential(n) * n).sum() / norm
        r2 = sum(x * x for x in _grid(self.n, self.h))
        got = {"norm": norm, "mu": kin + pot + contact + dipolar, "energy": kin + pot + 0.5 * (contact + dipolar), "kin": kin,
               "pot": pot, "contact": contact, "dipolar": dipolar, "rms_r": torch.sqrt((r2 * n).sum() / n.sum())}
        return {k: float(x) for k, x in got.items()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "sweep":
        problems, seeds = _sweep(case, seed)
        got = []
        for q, s in zip(problems, seeds):
            e = _Exact(q["n"], q["h"], q["nu"], q["gdd"], q["dt"], q["imag"], "xy")
            psi = _state(q["n"], q["h"], q["nu"], s)
            for _ in range(case["steps"]):
                psi = e.step(psi, q["g"])
            got.append(psi.cpu().numpy())
        return {"psi": got}
    n, h, nu = _axes(case)
    if kind == "potential":
        psi = _state(n, h, nu, seed).to(_dtype(case)).to(torch.complex128)
        e = _Exact(n, h, nu, 0.0, 1.0, True, case["kernel"])
        return e.potential(psi.real ** 2 + psi.imag ** 2)
    if kind == "gradient":
        psi, target, cm = _gradient_states(case, seed)
        e = _Exact(n, h, nu, case["gdd"], case["dt"], False, "dipolar3d")
        g = torch.tensor(case["g"], device="cuda", dtype=torch.float64, requires_grad=True)
        c = torch.tensor(cm, device="cuda", dtype=torch.float64, requires_grad=True)
        m = torch.arange(1, len(cm) + 1, device="cuda", dtype=torch.float64)
        for k in range(case["steps"]):
            psi = e.step(psi, g, 1.0 + (c * torch.sin(m * (k * case["dt"]))).sum())
        f = (math.prod(h) * (target.conj() * psi).sum()).abs() ** 2
        f.backward()
        return {"F": f.item(), "dg": g.grad.item(), "dc": [float(x) for x in c.grad]}
    e = _Exact(n, h, nu, case["gdd"], case["dt"], case["imag"], case["kernel"])
    psi = _run_state(case, seed).to(torch.complex128)
    for _ in range(case["steps"]):
        psi = e.step(psi, case["g"], strang=case["split"] == "strang")
    got = {"psi": psi}
    if case["observe"]:
        got.update(e.observe(psi, case["g"]))
    return got
